"""Register budgets of the kernels that the steps, the adjoint and the FV schemes
run, checked at build time (no GPU) on ptxas's resource report: what the comments
beside their launch bounds state, so that an added register does not cost a
resident CTA, or memory traffic of spills in every launch.

The report's names are mangled: template arguments in the order of the kernel's
declaration, n for a negative one."""
import re

import pytest

from test_kernel_resources import ptxas_report


def kernels(src, name):
    """{template arguments: report} of the kernels called name."""
    out = {}
    for entry, r in ptxas_report(src).items():
        m = re.match(rf"_ZN3cpr{len(name)}{name}I(.*?)EEv", entry)
        if m:
            args = re.findall(r"([fd]|L[ib]n?\d+E)", m.group(1) + "E")
            key = tuple(a if a in "fd" else int(a[2:-1].replace("n", "-")) for a in args)
            out[key] = r
    assert out, (src, name)
    return out


def resident(regs, threads):
    """CTAs per SM by registers (64 K, given out in eights per thread)."""
    return 65536 // ((regs + 7) // 8 * 8 * threads)


# resident CTAs per SM of the kernels for large grids of one problem, and threads per CTA
QUAD = {1: (7, 128), 2: (6, 192), 3: (4, 256), 4: (4, 160)}


@pytest.mark.parametrize("p", [1, 2, 3, 4])
def test_fp32_euler_stages(p):
    """cpr_stage_quad_kernel<P, DIV, FLUX, TX, TY, MINB, MODE>: for LP and Rusanov
    one kernel per stage mode, in a form for large grids and one for two CTAs per
    SM (p = 1 and 4: the same), none of which spills; the kernels for every mode
    (other divergences and fluxes, mode 0) spill only in the forms for large grids
    of p = 2 and 3, at most 48 bytes."""
    ctas, threads = QUAD[p]
    wide = ctas if p in (1, 4) else 2
    q = kernels(f"cpr_stage_f32_p{p}.cu", "cpr_stage_quad_kernel")
    modes = {}
    for (_, div, flux, _, _, minb, mode), r in q.items():
        if (div, flux) == (0, 0) and mode > 0:
            modes.setdefault(minb, set()).add(mode)
            assert r["spill"] == 0, (minb, mode, r)
            assert resident(r["regs"], threads) >= minb, (minb, mode, r)
        elif minb in (wide, ctas):
            assert r["spill"] <= (0 if minb == wide else 48), (div, flux, minb, r)
    assert {ctas, wide} == set(modes) and all(m == set(range(1, 7)) for m in modes.values()), modes


@pytest.mark.parametrize("p", [1, 2, 3, 4])
def test_fp32_adjoint(p):
    """cpr_vjp_quad_kernel: 8, 7, 5 and 4 tiles of 32 elements per SM, no spills."""
    (r,) = kernels(f"cpr_stage_f32_p{p}.cu", "cpr_vjp_quad_kernel").values()
    assert r["spill"] == 0 and resident(r["regs"], 32 * (p + 1)) >= {1: 8, 2: 7, 3: 5, 4: 4}[p], r


@pytest.mark.parametrize("p", [1, 2, 3, 4])
def test_fp64_euler_stages(p):
    """cpr_stage_f64_kernel<P, DIV, FLUX, TX, TY, MINB>: no spills; p = 3 keeps 16
    warps of 128 registers per SM."""
    for (_, div, flux, tx, ty, minb), r in kernels(f"cpr_stage_f64_p{p}.cu", "cpr_stage_f64_kernel").items():
        assert r["spill"] == 0, (div, flux, tx, ty, r)
        if p == 3:
            assert r["regs"] <= 128 and minb * 2 * tx * ty * 4 == 16 * 32, (div, flux, tx, ty, r)


@pytest.mark.parametrize("p", [1, 2, 3, 4])
@pytest.mark.parametrize("dtype", ["f32", "f64"])
def test_advection_stages(p, dtype):
    for key, r in kernels(f"cpr_stage_{dtype}_p{p}.cu", "cpr_stage_adv_kernel").items():
        assert r["spill"] == 0, (key, r)


def test_fv_stages():
    """cpr_fv_stage_kernel<T, EQ, FLUX, ORDER, MODE>: FP32 six CTAs of four warps
    (80 registers); only Roe's flux at third order spills, 12 bytes in the third
    stage.  FP64 twelve single warps or more."""
    for (_, eqn, flux, order, mode), r in kernels("cpr_fv_f32.cu", "cpr_fv_stage_kernel").items():
        assert r["regs"] <= 80, (eqn, flux, order, mode, r)
        assert r["spill"] <= (12 if (eqn, flux, order, mode) == (1, 2, 3, 6) else 0), (eqn, flux, order, mode, r)
    for key, r in kernels("cpr_fv_f32.cu", "cpr_fv_short_kernel").items():
        assert r["spill"] == 0 and r["regs"] <= 80, (key, r)
    for key, r in kernels("cpr_fv_f64.cu", "cpr_fv_stage_kernel").items():
        assert r["spill"] == 0 and resident(r["regs"], 32) >= 12, (key, r)
