"""Row chunks read in place, whose slope kernels run beside the MVM of the chunk before,
on the GPU: over many frames the commands are the whole-frame loop's bit for bit, with
two cameras, column blocks that end inside and at chunk ends, and a POLC product that
needs every command of the frame before; some frames are dropped after a few chunks."""
import numpy as np
import pytest

from paper_1903_01852_gb300 import synth
from parity_util import WAIT_US, device_frames

pytestmark = pytest.mark.gpu


def config(fmt, na, nblocks):
    from oracle import quantize_rows
    rng = np.random.default_rng(900 + na + nblocks)
    wfs = []
    for nsub, npx in ((40, 6), (22, 8)):
        w = synth.sh_wfs(rng, nsub, npx, nsub * npx, nsub * npx + 3, 0.2, ox=0, oy=0, nblocks=nblocks)
        wfs.append(w)
    ns = sum(2 * synth.num_valid(w) for w in wfs)
    M, P = synth.control_matrix(rng, na, ns, sd=1e-2), synth.polc_matrix(rng, na)
    ms = ps = None
    if fmt != "f32":
        (M, ms), (P, ps) = quantize_rows(M, fmt), quantize_rows(P, fmt)
    return dict(name="beside", na=na, ns=ns, wfs=wfs, M=M, M_scale=ms, M_dtype=fmt, P=P, P_scale=ps, P_dtype=fmt,
                gain=0.3, leak=0.05, clip=(-0.4, 0.4), a0=np.zeros(na, np.float32), ref_slopes=None)


def row_chunks(w, n):
    """Chunks of whole subaperture rows, the last to the end of the frame."""
    ends = [((k * w["nsuby"]) // n) * w["npx"] for k in range(1, n)] + [w["height"]]
    return list(zip([0] + ends[:-1], ends))


@pytest.mark.parametrize("where", ["host", "device"])
@pytest.mark.parametrize("fmt, na, nblocks, nchunks", [("f32", 700, 5, 5), ("f32", 3001, 3, 7), ("bf16", 700, 4, 10),
                                                       ("e4m3", 1500, 7, 4)])
def test_chunked_frames_equal_whole_ones_bitwise(rtc, where, fmt, na, nblocks, nchunks):
    torch = pytest.importorskip("torch")
    cfg = config(fmt, na, nblocks)
    frames = synth.draw_frames(cfg, 3, seed=901)
    dev = [device_frames(f) for f in frames]
    if where == "device":
        held = dev
    else:
        held = []
        for d in dev:                                       # page-locked, with the device frames' row pitch
            row = []
            for t in d:
                p = torch.empty((t.shape[0], t.stride(0)), dtype=torch.int16, pin_memory=True)
                p[:, :t.shape[1]] = t.cpu()
                row.append(p[:, :t.shape[1]])
            held.append(row)
    plans = [row_chunks(w, nchunks) for w in cfg["wfs"]]
    n = 40
    with rtc.Loop(cfg) as loop:
        want = []
        for k in range(n):
            loop.process_frame(k + 1, dev[k % 3])
            want.append(loop.get_commands(timeout_us=WAIT_US)[1])
    with rtc.Loop(cfg) as loop:
        fid = 0
        for k in range(n):
            if k % 7 == 3:                                  # a frame that never ends
                fid += 1
                for c in range(2):
                    for w, p in enumerate(plans):
                        loop.submit(fid, w, *p[c], held[(k + 1) % 3][w][p[c][0]:p[c][1]])
            fid += 1
            for c in range(nchunks):
                for w, p in enumerate(plans):
                    loop.submit(fid, w, *p[c], held[k % 3][w][p[c][0]:p[c][1]])
            got, a = loop.get_commands(timeout_us=WAIT_US)
            assert got == fid
            assert np.array_equal(a, want[k]), k
        assert loop.check_guards() == 0
