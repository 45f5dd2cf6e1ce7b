"""Frames written by the caller's own kernel on the loop's stream, on the GPU: the kernel
lets its dependents launch before it has written anything, and the frame must still be
the one it writes.  The commands are those of the same frames complete before the call,
bit for bit, with an implicit POLC (whose product would otherwise be the stream's last
kernel) and without."""
import ctypes as C
import subprocess

import numpy as np
import pytest

from paper_1903_01852_gb300 import build, synth
from parity_util import WAIT_US, device_frames

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def produce(tmp_path_factory):
    import os
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "stream_producer", "producer.cu")
    lib = str(tmp_path_factory.mktemp("producer") / "libproducer.so")
    subprocess.run([build.nvcc(), "-std=c++17", "-O2", *build.ARCH, "-shared", "-Xcompiler", "-fPIC", src, "-o", lib],
                   check=True)
    f = C.CDLL(lib).produce
    f.argtypes = [C.c_void_p, C.c_void_p, C.c_longlong, C.c_ulonglong, C.c_void_p]
    return f


@pytest.mark.parametrize("polc", [True, False])
@pytest.mark.parametrize("fmt", ["f32", "e4m3"])
def test_frames_written_on_the_loops_stream(rtc, produce, fmt, polc):
    torch = pytest.importorskip("torch")
    from oracle import quantize_rows
    rng = np.random.default_rng(950)
    w = synth.sh_wfs(rng, 24, 4, 104, 100, 0.1, nblocks=3)
    ns, na = 2 * synth.num_valid(w), 400
    M, P = synth.control_matrix(rng, na, ns, sd=1e-2), synth.polc_matrix(rng, na)
    ms = ps = None
    if fmt != "f32":
        (M, ms), (P, ps) = quantize_rows(M, fmt), quantize_rows(P, fmt)
    cfg = dict(name="caller", na=na, ns=ns, wfs=[w], M=M, M_scale=ms, M_dtype=fmt, P=P if polc else None,
               P_scale=ps if polc else None, P_dtype=fmt, gain=0.4, leak=0.02, clip=None,
               a0=rng.normal(0, 0.1, na).astype(np.float32), ref_slopes=None)
    source = [device_frames(f)[0] for f in synth.draw_frames(cfg, 6, seed=951)]
    want = []
    with rtc.Loop(cfg) as loop:
        for k, f in enumerate(source):
            loop.process_frame(k + 1, [f])
            want.append(loop.get_commands(timeout_us=WAIT_US)[1])
    got = []
    with rtc.Loop(cfg) as loop:
        stream = loop.stream()
        held = [torch.zeros(f.shape[0], f.stride(0), dtype=torch.int16, device="cuda") for f in source]
        torch.cuda.synchronize()
        for k in range(0, 6, 3):                            # three frames queued before their commands are read
            for j in range(k, k + 3):
                f = source[j]
                assert produce(held[j].data_ptr(), f.data_ptr(), f.shape[0] * f.stride(0), 100000, stream) == 0
                loop.process_frame(j + 1, [held[j][:, :f.shape[1]]])
            got += [loop.get_commands(timeout_us=WAIT_US)[1] for _ in range(3)]
    assert all(np.array_equal(a, b) for a, b in zip(got, want))
