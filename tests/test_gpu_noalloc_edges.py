"""rtc_reconstruct_noalloc around its kernel's steps (a lane's eight vectors of a split
of 1024 columns, the ragged end, warps of rows past the last), on the GPU, against
float64: |error| <= gamma_K (gain |scale| |M| |s|) + K u32 (the other terms), K the most
roundings on any path (one per column of the row at worst, and twelve after the sum)."""
import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

U32 = 2.0 ** -23


@pytest.mark.parametrize("ns", [1, 3, 4, 127, 128, 129, 1020, 1024, 1025, 2049, 4100])
@pytest.mark.parametrize("na", [1, 7, 9, 129])
def test_sizes_around_the_steps(rtc, na, ns):
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(10000 * na + ns)
    ld = (ns + 3) // 4 * 4 + 4
    M = np.full((na, ld), 7.0, np.float32)                  # the pitch is not read as part of the row
    M[:, :ns] = rng.standard_normal((na, ns))
    s, a, q = (rng.standard_normal(n).astype(np.float32) for n in (ns, na, na))
    scale = rng.uniform(0.5, 2.0, na).astype(np.float32)
    dev = [torch.from_numpy(x).cuda() for x in (M, scale, s, q, a)]
    sp = torch.zeros((ns + 3) // 4 * 4, device="cuda")
    sp[:ns] = dev[2]
    out = torch.empty(na, device="cuda")
    gain, leak = np.float32(0.45), np.float32(0.02)
    rc = rtc.lib.rtc_reconstruct_noalloc(na, ns, dev[0].data_ptr(), ld, dev[1].data_ptr(), sp.data_ptr(),
                                         dev[3].data_ptr(), dev[4].data_ptr(), out.data_ptr(), gain, leak,
                                         C.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert rc == rtc.RTC_OK
    torch.cuda.synchronize()
    m64, s64, a64, q64, c64 = (x.astype(np.float64) for x in (M[:, :ns], s, a, q, scale))
    oml = float(np.float32(1.0) - leak)
    want = float(gain) * (c64 * (m64 @ s64) + q64) + oml * a64
    K = ns + 12
    gamma = K * U32 / (1 - K * U32)
    bound = gamma * float(gain) * c64 * (np.abs(m64) @ np.abs(s64)) + 12 * U32 * (np.abs(q64) + np.abs(a64))
    assert np.all(np.abs(out.cpu().numpy() - want) <= bound)
