"""E4M3 and BF16 matrices at the edges of the product kernels' lane groups, on the GPU.

An E4M3 row is stored in groups of 16 vectors of 16 codes (the last group shorter), in
an order of its own; the POLC products take whole steps of several groups first.  Column
counts on both sides of a vector, a group and a step, and row counts on both sides of a
warp's rows, against the FP64 oracle at the repository's float32 tolerance: the products
are exact in float32 and only their sums round, as for a float32 matrix."""
import numpy as np
import pytest

from oracle import quantize_rows
from paper_1903_01852_gb300 import synth
from parity_util import WAIT_US, device_frames, run_pair

pytestmark = pytest.mark.gpu


def lane_config(units, na, fmt, nblocks, seed):
    """One SH sensor of 24 x 24 subapertures, the first `units` of them valid."""
    rng = np.random.default_rng(seed)
    w = synth.sh_wfs(rng, 24, 2, 50, 48, 0.0, nblocks=nblocks)
    w["valid"] = (np.arange(24 * 24) < units).reshape(24, 24)
    ns = 2 * units
    M, ms = quantize_rows(synth.control_matrix(rng, na, ns, sd=1e-2), fmt)
    P, ps = quantize_rows(synth.polc_matrix(rng, na), fmt)
    return dict(name="lanes", na=na, ns=ns, wfs=[w], M=M, M_scale=ms, M_dtype=fmt, P=P, P_scale=ps, P_dtype=fmt,
                gain=0.45, leak=0.02, clip=None, a0=rng.normal(0, 0.1, na).astype(np.float32),
                ref_slopes=rng.normal(0, 0.1, ns).astype(np.float32))


@pytest.mark.parametrize("fmt", ["e4m3", "bf16"])
@pytest.mark.parametrize("units", [1, 7, 8, 9, 120, 128, 129, 248, 256, 257, 384, 512, 513, 576])
def test_column_counts_around_lane_groups(rtc, units, fmt):
    pytest.importorskip("torch")
    cfg = lane_config(units, 33, fmt, 1, seed=400 + units)
    frames = synth.draw_frames(cfg, 2, seed=401)
    with rtc.Loop(cfg, telemetry=True) as loop:
        run_pair(loop, cfg, frames, mode="whole")


@pytest.mark.parametrize("fmt", ["e4m3", "bf16"])
@pytest.mark.parametrize("na", [1, 2, 3, 31, 767, 768, 769, 1023, 1024, 1025, 1040])
def test_row_counts_and_polc_steps(rtc, na, fmt):
    pytest.importorskip("torch")
    cfg = lane_config(200, na, fmt, 3, seed=500 + na)
    frames = synth.draw_frames(cfg, 3, seed=501)
    with rtc.Loop(cfg, telemetry=True) as loop:
        _, chunked = run_pair(loop, cfg, frames, nchunks=3)
    with rtc.Loop(cfg, telemetry=True) as loop:
        _, whole = run_pair(loop, cfg, frames, mode="whole")
    assert all(np.array_equal(a, b) for a, b in zip(chunked, whole))


@pytest.mark.parametrize("units", [9, 129, 300])
def test_updated_matrices_equal_uploaded_ones_bitwise(rtc, units):
    pytest.importorskip("torch")
    cfg = lane_config(units, 300, "e4m3", 2, seed=600)
    other = lane_config(units, 300, "e4m3", 2, seed=601)
    cfg["a0"][:] = 0                       # the first frame's POLC term, P a0, is then the same with either P
    matrices = {k: other[k] for k in ("M", "M_scale", "P", "P_scale")}
    frames = [device_frames(f) for f in synth.draw_frames(cfg, 3, seed=602)]

    def commands(loop):
        out = []
        for k, f in enumerate(frames):
            loop.process_frame(k + 1, f)
            out.append(loop.get_commands(timeout_us=WAIT_US)[1])
        return out

    with rtc.Loop(dict(cfg, **matrices)) as loop:
        want = commands(loop)
    with rtc.Loop(cfg, updatable=True) as loop:
        for _ in range(2):                 # the second goes into buffers that the first has put in order
            loop.update(**matrices)
        got = commands(loop)
    assert all(np.array_equal(a, b) for a, b in zip(got, want))
