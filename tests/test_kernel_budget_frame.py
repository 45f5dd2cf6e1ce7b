"""Register and spill budgets (as test_kernel_budget, CPU only) of the kernels whose loads
in flight and resident CTAs set their speed: the float32 MVM of large whole frames, the
narrow formats' launches of few CTAs, the finalisation, the quantiser, and
rtc_reconstruct_noalloc."""
import os

import test_kernel_budget as base

# mangled entry -> (what, register budget, spill budget in bytes)
KERNELS = {
    # five CTAs of 256 threads per SM at 48 registers
    "_ZN3rtc16gemv_kernel_wideILi1EEEvNS_8GemvArgsE": ("float32 whole-frame MVM, 1 row per warp", 48, 0),
    "_ZN3rtc16gemv_kernel_wideILi4EEEvNS_8GemvArgsE": ("float32 whole-frame MVM, 4 rows per warp", 48, 0),
    # two CTAs per SM at 128; plain and pre-enqueued
    **{f"_ZN3rtc16gemv_kernel_deepILi{dt}ELi{u}ELi{ri}ELb{g}EEEvNS_8GemvArgsE": (f"{what} launch of few CTAs", 128, 0)
       for dt, u, what in ((1, 3, "BF16"), (2, 2, "E4M3")) for ri in (2, 4) for g in (0, 1)},
    "_ZN3rtc15finalise_kernelENS_12FinaliseArgsEPKfi": ("finalisation", 32, 0),
    "_ZN3rtc16normalise_kernelENS_8NormArgsE": ("pyramid normalisation", 32, 0),
    # the CTAs per SM of quantize_kernel's bounds
    **{f"_ZN3rtc15quantize_kernelILi{dt}ELi{t}ELi{c}EEEviPKfmPvPf": (f"quantiser, {t} threads", r, 0)
       for dt in (1, 2) for t, c, r in ((64, 24, 40), (128, 12, 40), (256, 6, 40), (512, 3, 40), (1024, 2, 32))},
}
# anonymous namespace: looked up by the end of the name
NOALLOC = {"17split_gemv_kernelEPKfmiiiS1_Pf": ("split MVM, five CTAs per SM", 48, 16),
           "21split_finalise_kernelEPKfiiS1_S1_S1_Pfff": ("split finalisation", 32, 0)}


def check(report, name, what, regs, spill):
    assert name in report, f"{what}: entry {name} not compiled"
    assert report[name]["regs"] <= regs, f"{what}: {report[name]['regs']} registers > {regs}"
    assert report[name].get("spill", 0) <= spill, f"{what}: {report[name]['spill']} bytes of spill > {spill}"


def test_frame_kernels_stay_within_their_register_budget():
    report = base.ptxas_report()
    for name, budget in KERNELS.items():
        check(report, name, *budget)


def test_noalloc_kernels_stay_within_their_register_budget(monkeypatch):
    monkeypatch.setattr(base, "SRC", os.path.join(os.path.dirname(base.SRC), "rtc_noalloc.cu"))
    report = base.ptxas_report()
    for end, budget in NOALLOC.items():
        names = [n for n in report if n.endswith(end)]
        assert len(names) == 1, end
        check(report, names[0], *budget)
