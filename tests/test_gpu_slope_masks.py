"""Shack-Hartmann rows of which the slope kernel reads only the quads of four pixels from
the first to the last valid subaperture, without its widest gap: masks whose ends and
gaps fall on and off quad boundaries, for offsets 0 to 3 and odd subaperture sizes,
against the FP64 oracle at the repository's float32 tolerance, whole and in chunks."""
import numpy as np
import pytest

from paper_1903_01852_gb300 import synth
from parity_util import run_pair

pytestmark = pytest.mark.gpu


def masks(n):
    rows = np.zeros((n, n), bool)
    rows[0, :] = True                       # full row
    rows[1, 0] = True                       # one unit at either end, or inside
    rows[2, n - 1] = True
    rows[3, n // 2] = True
    rows[4, [0, n - 1]] = True              # the widest gap there is
    rows[5, ::2] = True                     # gaps of one
    rows[6, [1, 2, 5, n - 2]] = True        # two gaps, the second wider
    rows[7, [0, 4, 5, n - 3]] = True
    return rows                             # the last rows have no valid unit


@pytest.mark.parametrize("ox", [0, 1, 2, 3])
@pytest.mark.parametrize("npx", [2, 3, 5, 8])
def test_masked_rows(rtc, npx, ox):
    pytest.importorskip("torch")
    rng = np.random.default_rng(10 * npx + ox)
    n = 11
    w = synth.sh_wfs(rng, n, npx, n * npx + 7, n * npx + 5, 0.0, ox=ox, oy=2, nblocks=3)
    w["valid"] = masks(n)
    ns, na = 2 * int(w["valid"].sum()), 19
    cfg = dict(name="masks", na=na, ns=ns, wfs=[w], M=synth.control_matrix(rng, na, ns, sd=1e-2), M_scale=None, M_dtype="f32",
               P=None, P_scale=None, P_dtype="f32", gain=0.4, leak=0.02, clip=None, a0=np.zeros(na, np.float32),
               ref_slopes=rng.normal(0, 0.1, ns).astype(np.float32))
    frames = synth.draw_frames(cfg, 2, seed=801)
    for mode in ("whole", "chunked"):
        with rtc.Loop(cfg, telemetry=True) as loop:
            run_pair(loop, cfg, frames, mode=mode, nchunks=4)
