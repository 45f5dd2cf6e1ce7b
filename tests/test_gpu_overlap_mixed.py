"""One implicit-POLC loop whose frames arrive in turn whole, in row chunks read in place
and as graph launches, three at a time before anything is read back, with parameter
updates between them: a frame's slopes start beside the POLC product of the frame before
(whichever way that came), beside the MVM of the chunk before, or after a graph.
Commands and telemetry slopes are the bits of a loop whose timing events keep every
launch apart."""
import numpy as np
import pytest

from paper_1903_01852_gb300 import synth
from parity_util import WAIT_US, device_frames

pytestmark = pytest.mark.gpu

N = 36


def config(fmt, nsub, na, nblocks, seed=960):
    from oracle import quantize_rows
    rng = np.random.default_rng(seed)
    wfs = [synth.sh_wfs(rng, nsub, 4, 4 * nsub + 4, 4 * nsub, 0.15, ox=0, oy=0, nblocks=nblocks),
           synth.sh_wfs(rng, 9, 6, 60, 54, 0.0, ox=0, oy=0, nblocks=2)]
    ns = sum(2 * synth.num_valid(w) for w in wfs)
    M, P = synth.control_matrix(rng, na, ns, sd=1e-2), synth.polc_matrix(rng, na)
    ms = ps = None
    if fmt != "f32":
        (M, ms), (P, ps) = quantize_rows(M, fmt), quantize_rows(P, fmt)
    return dict(name="mixed", na=na, ns=ns, wfs=wfs, M=M, M_scale=ms, M_dtype=fmt, P=P, P_scale=ps, P_dtype=fmt,
                gain=0.4, leak=0.03, clip=(-0.5, 0.5), a0=rng.normal(0, 0.1, na).astype(np.float32),
                ref_slopes=rng.normal(0, 0.05, ns).astype(np.float32))


def pinned(torch, dev):
    out = []
    for t in dev:
        p = torch.empty((t.shape[0], t.stride(0)), dtype=torch.int16, pin_memory=True)
        p[:, :t.shape[1]] = t.cpu()
        out.append(p[:, :t.shape[1]])
    return out


def row_chunks(w, n):
    ends = [((k * w["nsuby"]) // n) * w["npx"] for k in range(1, n)] + [w["height"]]
    return list(zip([0] + ends[:-1], ends))


def updates(cfg, other, k):
    """The parameters that change before frame k, or None."""
    if k % 6 != 4:                          # the frame before is still queued
        return None
    src = other if k % 12 == 4 else cfg
    return {key: src[key] for key in ("M", "M_scale", "P", "P_scale", "ref_slopes") if src[key] is not None}


def run(rtc, cfg, other, frames, dev, host, modes, **kw):
    plans = [row_chunks(w, 5) for w in cfg["wfs"]]
    out = []
    with rtc.Loop(cfg, telemetry=True, ring=6, **kw) as loop:
        for k in range(N):
            new = updates(cfg, other, k) if other else None
            if new:
                loop.update(**new)
            mode = modes[k % len(modes)]
            if mode == "whole":
                loop.process_frame(k + 1, dev[k % 4])
            elif mode == "host":
                loop.process_frame(k + 1, host[k % 4])
            elif mode == "chunks":
                for c in range(5):
                    for i, p in enumerate(plans):
                        loop.submit(k + 1, i, *p[c], host[k % 4][i][p[c][0]:p[c][1]])
            else:
                for buf, frame in zip(loop.next_frame_buffers(), frames[k % 4]):
                    buf[:] = frame
                loop.submit_graph(k + 1)
            if k % 3 == 2:
                for j in range(k - 1, k + 2):
                    fid, a = loop.get_commands(timeout_us=WAIT_US)
                    assert fid == j
                    out.append((a, loop.get_telemetry(fid, timeout_us=WAIT_US)[0]))
        assert loop.check_guards() == 0
    return out


@pytest.mark.parametrize("fmt, nsub, na, nblocks", [("f32", 40, 900, 4), ("f32", 80, 1200, 6), ("bf16", 40, 900, 5),
                                                    ("e4m3", 60, 2000, 8)])
@pytest.mark.parametrize("way", ["updates", "graphs"])
def test_mixed_frames(rtc, way, fmt, nsub, na, nblocks):
    torch = pytest.importorskip("torch")
    cfg, other = config(fmt, nsub, na, nblocks), config(fmt, nsub, na, nblocks, seed=961)
    if way == "graphs":                     # a loop with graphs takes no updates
        other, kw = None, dict(graphs=True)
        modes = ["graph", "whole", "chunks", "whole", "host", "graph", "chunks"]
    else:
        kw = dict(updatable=True)
        modes = ["whole", "whole", "chunks", "host", "chunks", "chunks", "whole"]
    frames = synth.draw_frames(cfg, 4, seed=962)
    dev = [device_frames(f) for f in frames]
    host = [pinned(torch, d) for d in dev]
    want = run(rtc, cfg, other, frames, dev, host, ["whole"], timing=True, updatable=other is not None)
    got = run(rtc, cfg, other, frames, dev, host, modes, **kw)
    assert len(want) == len(got) == N
    for k, ((a, s), (b, t)) in enumerate(zip(got, want)):
        assert np.array_equal(a, b) and np.array_equal(s, t), (k, modes[k % len(modes)])
