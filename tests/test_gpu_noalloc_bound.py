"""rtc_reconstruct_noalloc against float64 with a bound of its own summation path, at the
sizes of its steps.

A row is cut into splits of at most 1024 columns.  A lane adds two products of each of its
float4 vectors to either of two sums (v vectors: 2 v fused multiply-adds on a path), the
two sums, at most one column of the ragged end, then come five steps over the lanes, the
sum of the splits, the row scale, q and the gain.  So the product terms see at most
K = 2 v + 1 + 1 + 5 + nsplit + 3 roundings of 2^-24, q and a (with its product by
1 - leak) two each.  The same inputs with the matrix rounded to BF16, and with any one
column left out, lie outside the bound at every size (checked here, on the CPU)."""
import ctypes as C

import numpy as np
import pytest

U = 2.0 ** -24
NS = [1, 3, 4, 127, 128, 129, 1020, 1024, 1025, 2049, 4100, 8608]
NA = [1, 7, 9, 129]
GAIN, LEAK = np.float32(0.45), np.float32(0.02)


def inputs(na, ns):
    rng = np.random.default_rng(20000 * na + ns)
    away = lambda *n: (rng.uniform(0.25, 2.0, n) * rng.choice([-1.0, 1.0], n)).astype(np.float32)  # noqa: E731
    return away(na, ns), away(ns), away(na), away(na), rng.uniform(0.5, 2.0, na).astype(np.float32)


def exact_and_bound(M, s, q, a, scale):
    m64, s64, q64, a64, c64 = (x.astype(np.float64) for x in (M, s, q, a, scale))
    oml, gain = float(np.float32(1.0) - LEAK), float(GAIN)
    ns = len(s)
    nsplit = -(-ns // 1024)
    cols = -(-ns // nsplit)
    cols = -(-cols // 4) * 4
    nsplit = -(-ns // cols)
    K = 2 * -(-(cols // 4) // 32) + 1 + 1 + 5 + nsplit + 3
    gamma = lambda k: k * U / (1 - k * U)  # noqa: E731
    y = c64 * (m64 @ s64)
    bound = gamma(K) * gain * c64 * (np.abs(m64) @ np.abs(s64)) + gamma(2) * (gain * np.abs(q64) + oml * np.abs(a64))
    return gain * (y + q64) + oml * a64, bound


@pytest.mark.parametrize("ns", NS)
@pytest.mark.parametrize("na", NA)
def test_the_bound_tells_a_rounded_matrix_and_a_lost_column(na, ns):
    M, s, q, a, scale = inputs(na, ns)
    want, bound = exact_and_bound(M, s, q, a, scale)
    bits = M.view(np.uint32)                                # round to nearest even at 16 bits: BF16
    bf16 = ((bits + 0x7FFF + ((bits >> 16) & 1)) & np.uint32(0xFFFF0000)).view(np.float32)
    assert np.any(np.abs(exact_and_bound(bf16, s, q, a, scale)[0] - want) > 2 * bound)
    term = float(GAIN) * scale[:, None].astype(np.float64) * np.abs(M * s.astype(np.float64))
    assert np.all(term > 2 * bound[:, None])


@pytest.mark.gpu
@pytest.mark.parametrize("ns", NS)
@pytest.mark.parametrize("na", NA)
def test_error_within_the_bound_of_its_sums(rtc, na, ns):
    torch = pytest.importorskip("torch")
    M, s, q, a, scale = inputs(na, ns)
    want, bound = exact_and_bound(M, s, q, a, scale)
    ld = (ns + 3) // 4 * 4
    wide = np.full((na, ld), 7.0, np.float32)               # the pitch is not read as part of the row
    wide[:, :ns] = M
    sp = np.full(ld, 7.0, np.float32)
    sp[:ns] = s
    dev = [torch.from_numpy(x).cuda() for x in (wide, scale, sp, q, a)]
    out = torch.empty(na, device="cuda")
    rc = rtc.lib.rtc_reconstruct_noalloc(na, ns, dev[0].data_ptr(), ld, *(d.data_ptr() for d in dev[1:]), out.data_ptr(),
                                         GAIN, LEAK, C.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert rc == rtc.RTC_OK
    torch.cuda.synchronize()
    assert np.all(np.abs(out.cpu().numpy() - want) <= bound)
