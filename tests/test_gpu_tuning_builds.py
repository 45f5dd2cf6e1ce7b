"""Builds with other values of the kernels' tuning macros, on the GPU: whole and chunked
frames give the same bits and the FP64 oracle's commands to the float32 tolerance."""
import os
import subprocess
import sys
import textwrap

import pytest

pytestmark = pytest.mark.gpu

SCRIPT = textwrap.dedent("""
    import sys, numpy as np
    sys.path.insert(0, "tests")
    from oracle import OracleLoop, quantize_rows
    from paper_1903_01852_gb300 import binding as rtc, synth
    from parity_util import TOL_F32, WAIT_US, device_frames, rel
    from test_gpu_whole_frame import config
    fmt, nsub, na, nblocks = sys.argv[1], *map(int, sys.argv[2:5])
    cfg = config(nsub, na, nblocks)
    if fmt != "f32":
        (m, ms), (p, ps) = quantize_rows(cfg["M"], fmt), quantize_rows(cfg["P"], fmt)
        cfg.update(M=m, M_scale=ms, M_dtype=fmt, P=p, P_scale=ps, P_dtype=fmt)
    ref = OracleLoop(cfg)
    with rtc.Loop(cfg) as whole, rtc.Loop(cfg) as chunked:
        for k, f in enumerate(synth.draw_frames(cfg, 2, seed=703)):
            whole.process_frame(k + 1, device_frames(f))
            chunked.submit_frame(k + 1, f, [synth.chunk_plan(w, 4) for w in cfg["wfs"]])
            a, b = (x.get_commands(timeout_us=WAIT_US)[1] for x in (whole, chunked))
            assert np.array_equal(a, b), k
            assert rel(a, ref.step(f)[1]) <= TOL_F32, k
    print("ok")
""")


def run_with(defines, tmp_path, cases):
    from paper_1903_01852_gb300.build import build
    pytest.importorskip("torch")
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    lib = build(defines=defines, out=str(tmp_path / "librtc.so"))
    env = dict(os.environ, RTC_LIBRARY=lib, PYTHONPATH=root + os.pathsep + os.environ.get("PYTHONPATH", ""))
    for case in cases:
        r = subprocess.run([sys.executable, "-c", SCRIPT, *map(str, case)], env=env, capture_output=True, text=True,
                           timeout=600, cwd=root)
        assert r.returncode == 0 and r.stdout.startswith("ok"), (case, r.stdout[-2000:] + r.stderr[-3000:])


def test_float32_sums_of_one_fma_per_element(tmp_path):
    # without packed sums a launch may take two rows per warp: whole frames of 50000 rows x blocks, rows of 160 vectors
    run_with(["RTC_GEMV_FFMA2_MASK=0"], tmp_path, [("f32", 80, 2500, 20), ("f32", 24, 240, 3)])


@pytest.mark.parametrize("lanes", [16, 32])
def test_packed_sums_of_the_narrow_formats(tmp_path, lanes):
    # few-CTA launches (four and two rows per warp), grouped whole frames, rows of one vector to 50
    cases = [(fmt, *size) for fmt in ("e4m3", "bf16") for size in ((24, 200, 3), (6, 33, 5), (40, 2500, 4))]
    run_with(["RTC_GEMV_FFMA2_MASK=7", f"RTC_GEMV_E4M3_LANES={lanes}"], tmp_path, cases + [("e4m3", 60, 6000, 28)])
