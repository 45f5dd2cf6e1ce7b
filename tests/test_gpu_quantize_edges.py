"""rtc_quantize_rows at the edges of its kernels, on the GPU: codes and scales are the
oracle's bit for bit (so no tolerance) for row lengths on both sides of each choice of
threads, rows off the 16-byte boundary, rows with a pitch, quotients on and next to the
boundary between two codes, scales and quotients near the ends of the float32 range."""
import numpy as np
import pytest

from oracle import quantize_rows

pytestmark = pytest.mark.gpu

U = {"bf16": np.uint16, "e4m3": np.uint8}


def gpu_codes(rtc, M, fmt):
    torch = pytest.importorskip("torch")
    codes, scale = rtc.quantize_rows(M, fmt)
    torch.cuda.synchronize()
    return codes.cpu().numpy().view(U[fmt]), scale.cpu().numpy()


@pytest.mark.parametrize("fmt", ["bf16", "e4m3"])
@pytest.mark.parametrize("offset", [0, 1, 3])
@pytest.mark.parametrize("ns", [1, 2, 3, 4, 5, 7, 255, 1535, 1536, 6999, 7001, 18000, 34001, 40003])
def test_row_lengths_offsets_and_pitches(rtc, ns, offset, fmt):
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(ns + offset)
    base = (rng.standard_normal((5, ns + offset)) * 10.0 ** rng.uniform(-6, 6, (5, 1))).astype(np.float32)
    M = base[:, offset:]
    codes, scale = gpu_codes(rtc, torch.from_numpy(base).cuda()[:, offset:], fmt)
    c_ref, s_ref = quantize_rows(np.ascontiguousarray(M), fmt)
    assert np.array_equal(scale, s_ref)
    assert np.array_equal(codes, c_ref)


@pytest.mark.parametrize("fmt", ["bf16", "e4m3"])
def test_quotients_at_code_boundaries_and_range_ends(rtc, fmt):
    torch = pytest.importorskip("torch")
    # every value half way between two codes of the format, its float32 neighbours, both signs
    if fmt == "e4m3":
        mant, exps = np.arange(16, 32) / 16.0, np.arange(-9, 9)
    else:
        mant, exps = np.arange(256, 512) / 256.0, np.arange(-12, 1)
    mid = np.unique(np.concatenate([m * 2.0 ** exps for m in mant] + [np.arange(0, 17) * 2.0 ** -10]))
    mid = mid.astype(np.float32)
    vals = np.concatenate([mid, np.nextafter(mid, np.float32(0)), np.nextafter(mid, np.float32(np.inf))])
    vals = np.concatenate([vals, -vals, np.float32([1e-38, -1e-38, 1e-42, -1e-45, 0.0, -0.0])])
    rows = []
    top = np.float32(448.0 if fmt == "e4m3" else 2.0)
    for scale in (1.0, 3.0, 0.7, 1e-3, 1e-33, 1e-38, 1e33, 7e35):
        with np.errstate(under="ignore"):
            r = np.minimum(np.maximum(vals, -top), top) * np.float32(scale)
        rows.append(np.concatenate([r, [top * np.float32(scale)]]).astype(np.float32))
    M = np.stack(rows)
    codes, scale = gpu_codes(rtc, torch.from_numpy(M).cuda(), fmt)
    c_ref, s_ref = quantize_rows(M, fmt)
    assert np.array_equal(scale, s_ref)
    assert np.array_equal(codes, c_ref)


def test_rows_with_nan_and_inf(rtc):
    # a NaN does not count in a row's maximum and gets the NaN code; beside an infinity
    # (scale inf) finite elements get the code of a zero, infinities that of a NaN
    torch = pytest.importorskip("torch")
    M = np.float32([[np.nan, 448.0, -224.0, 0.0, 1.0], [np.inf, -2.0, 3.0, -np.inf, 0.0], [np.nan] * 5])
    codes, scale = gpu_codes(rtc, torch.from_numpy(M).cuda(), "e4m3")
    assert np.array_equal(scale, np.float32([1.0, np.inf, 1.0]))
    assert codes[0].tolist() == [0x7F, 0x7E, 0xF6, 0x00, 0x38]
    assert codes[1].tolist() == [0x7F, 0x80, 0x00, 0x7F, 0x00]
    assert codes[2].tolist() == [0x7F] * 5
    codes, scale = gpu_codes(rtc, torch.from_numpy(M).cuda(), "bf16")
    assert np.array_equal(scale, np.float32([448.0, np.inf, 1.0]))
    assert codes[0].tolist() == [0x7FFF, 0x3F80, 0xBF00, 0x0000, 0x3B12]
    assert codes[1].tolist() == [0x7FFF, 0x8000, 0x0000, 0x7FFF, 0x0000]
    assert codes[2].tolist() == [0x7FFF] * 5
