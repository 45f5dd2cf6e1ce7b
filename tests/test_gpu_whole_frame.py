"""Whole-frame launches whose finalisation is a kernel of its own, on the GPU.

From 1 MB of float32 matrix on, a whole frame's MVM leaves its finalisation to a
dependent kernel, and rows of more than 128 vectors go to a kernel of their own; a frame
that arrives in row chunks finalises in the tail of its launches.  Every row's sum and
every finalisation keeps its order, so the commands are the same bits, on both sides of
each rule (and, at the smaller sizes, the oracle's to the float32 tolerance)."""
import numpy as np
import pytest

from oracle import OracleLoop
from paper_1903_01852_gb300 import synth
from parity_util import TOL_F32, WAIT_US, device_frames, rel

pytestmark = pytest.mark.gpu


def config(nsub, na, nblocks, clip=None, polc=True):
    rng = np.random.default_rng(7000 + nsub + na + nblocks)
    w = synth.sh_wfs(rng, nsub, 2, 2 * nsub + 2, 2 * nsub, 0.0, nblocks=nblocks)
    w["valid"] = np.ones((nsub, nsub), bool)
    ns = 2 * nsub * nsub
    return dict(name="whole", na=na, ns=ns, wfs=[w], M=synth.control_matrix(rng, na, ns, sd=1e-2), M_scale=None,
                M_dtype="f32", P=synth.polc_matrix(rng, na) if polc else None, P_scale=None, P_dtype="f32",
                gain=0.45, leak=0.02, clip=clip, a0=rng.normal(0, 0.1, na).astype(np.float32), ref_slopes=None)


# (subapertures across, rows, column blocks): 0.9 MB fused; 1.1 MB separate, one block; rows of 128 and of 129
# vectors; one row per warp; four rows per warp of 133 vectors
@pytest.mark.parametrize("nsub, na, nblocks", [(24, 200, 3), (24, 240, 1), (16, 1000, 1), (23, 1001, 2), (24, 2049, 2),
                                               (80, 3300, 24)])
def test_whole_frames_equal_chunked_ones_bitwise(rtc, nsub, na, nblocks):
    pytest.importorskip("torch")
    big = na * nsub > 100000
    cfg = config(nsub, na, nblocks, clip=(-0.3, 0.3), polc=not big)
    frames = synth.draw_frames(cfg, 3, seed=701)
    plans = [synth.chunk_plan(w, 4) for w in cfg["wfs"]]
    got = {}
    for mode in ("chunks", "whole", "graph"):
        with rtc.Loop(cfg, graphs=mode == "graph") as loop:
            out = []
            for k, f in enumerate(frames):
                if mode == "chunks":
                    loop.submit_frame(k + 1, f, plans)
                elif mode == "whole":
                    loop.process_frame(k + 1, device_frames(f))
                else:
                    for buf, frame in zip(loop.next_frame_buffers(), f):
                        buf[:] = frame
                    loop.submit_graph(k + 1)
                out.append(loop.get_commands(timeout_us=WAIT_US)[1])
            assert loop.check_guards() == 0
            got[mode] = out
    for mode in ("whole", "graph"):
        assert all(np.array_equal(a, b) for a, b in zip(got["chunks"], got[mode])), mode
    if not big:
        ref = OracleLoop(cfg)
        for a, f in zip(got["whole"], frames):
            assert rel(a, ref.step(f)[1]) <= TOL_F32


@pytest.mark.parametrize("fmt, nsub, na, nblocks", [("f32", 24, 200, 3), ("f32", 40, 1001, 4), ("bf16", 40, 2500, 4),
                                                    ("e4m3", 40, 2500, 8)])
def test_frames_in_a_row_start_beside_the_polc_product(rtc, fmt, nsub, na, nblocks):
    # With an implicit POLC a frame's slopes run beside the POLC product of the frame before.  Frames submitted
    # three at a time before their commands are read, with and without slope telemetry, against a loop whose
    # timing events keep them apart.
    pytest.importorskip("torch")
    from oracle import quantize_rows
    cfg = config(nsub, na, nblocks, clip=(-0.3, 0.3))
    if fmt != "f32":
        (m, ms), (p, ps) = quantize_rows(cfg["M"], fmt), quantize_rows(cfg["P"], fmt)
        cfg.update(M=m, M_scale=ms, M_dtype=fmt, P=p, P_scale=ps, P_dtype=fmt)
    frames = [device_frames(f) for f in synth.draw_frames(cfg, 5, seed=702)]
    want = []
    with rtc.Loop(cfg, timing=True) as loop:
        for k in range(30):
            loop.process_frame(k + 1, frames[k % 5])
            want.append(loop.get_commands(timeout_us=WAIT_US)[1])
    for telemetry in (False, True):
        with rtc.Loop(cfg, telemetry=telemetry) as loop:
            for k in range(0, 30, 3):
                for j in range(3):
                    loop.process_frame(k + j + 1, frames[(k + j) % 5])
                for j in range(3):
                    fid, a = loop.get_commands(timeout_us=WAIT_US)
                    assert fid == k + j + 1 and np.array_equal(a, want[k + j]), (telemetry, k + j)
            assert loop.check_guards() == 0
