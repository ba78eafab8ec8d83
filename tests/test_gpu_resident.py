"""The linear solve with the matrix resident in shared memory (one cooperative launch) against the
same solve as separate kernels (BHEM_PCG_LOOP=host), at the edges of its dispatch: one to 34 rows
per CTA in FP32 and one to 17 in FP64 (152 SMs), each register form's last and first row count, the
first size that no longer fits, periodic grids, masks, negative curvature and an expired wait.

Tolerances. Both forms run block-Jacobi PCG on the same matrix from the same start; sums over a row
and over the grid, and the block inverses, are rounded differently, so iteration counts agree within
one and the solutions to what the stopping rule leaves, |r| <= rtol |b|: 1e-4 relative for mixed
precision at rtol 1e-6 (as for the other single-launch forms), and for FP64 at rtol 1e-12 the same
ratio, 1e-10 (the block-Jacobi-scaled systems here, M / dt^2 + K with dt = 1 ms, have condition
numbers below 100)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2312_14839_gb300 import scenes as S  # noqa: E402

pytestmark = pytest.mark.gpu


def dev(a, dtype=torch.float64):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=dtype, device="cuda")


def state(shape, nu, nv):
    if shape == "annulus":
        g, rest = S.annulus(nu, nv)
        side = 0.2 * g.dxi1
    else:
        g, rest = S.flat_sheet(nu, nv, nu / max(nu, nv), nv / max(nu, nv))
        side = g.dxi1
    return g, rest, S.noisy(rest, 3e-3 * min(side, g.dxi2), 5)


def solve(monkeypatch, form, g, rest, q, prec, mask, rtol, fixed=0, mass_scale=1e6):
    from paper_2312_14839_gb300.bhem import Shell
    if form is None:
        monkeypatch.delenv("BHEM_PCG_LOOP", raising=False)
    else:
        monkeypatch.setenv("BHEM_PCG_LOOP", form)
    with Shell(g, S.SHEET_MATERIAL, dev(rest.reshape(-1)), precision=prec, assembly="color") as sh:
        _, G = sh.energy_grad_hess(dev(q.reshape(-1)), mass_scale=mass_scale)
        n0 = sh.kernel_launches()
        x, it, neg = sh.pcg_solve(-G, mask=mask, rtol=rtol, max_iter=2000, fixed_iters=fixed)
        x2, it2, _ = sh.pcg_solve(-G, mask=mask, rtol=rtol, max_iter=2000, fixed_iters=fixed)
        assert it2 == it and torch.equal(x, x2)   # deterministic
        return x.cpu().numpy(), it, neg, (sh.kernel_launches() - n0) // 2


@pytest.mark.parametrize("shape,nu,nv,prec,resident", [
    ("sheet", 1, 1, "mixed", True), ("sheet", 1, 1, "fp64", True),          # 4 nodes: one CTA
    ("annulus", 2, 1, "mixed", True), ("annulus", 2, 1, "fp64", True),      # every row couples to all
    ("annulus", 7, 2, "mixed", True), ("annulus", 7, 2, "fp64", True),
    ("sheet", 10, 10, "mixed", True), ("sheet", 10, 10, "fp64", True),
    ("sheet", 35, 37, "mixed", True),      # 1,368 nodes: 9 rows per CTA on 152 SMs
    ("sheet", 36, 36, "mixed", True),      # 1,369: 10
    ("annulus", 280, 5, "mixed", True),    # 1,680: 12, the last CTA short
    ("sheet", 46, 46, "mixed", True),      # 2,209: 15
    ("sheet", 52, 52, "mixed", True),      # 2,809: 19
    ("sheet", 64, 64, "mixed", True),      # 4,225: 28
    ("sheet", 65, 65, "mixed", True),      # 4,356: 29, matrix read from shared memory
    ("sheet", 72, 71, "mixed", False),     # 5,256: 35 rows do not fit
    ("sheet", 35, 37, "fp64", True),       # 9
    ("sheet", 36, 36, "fp64", True),       # 10: from shared memory
    ("sheet", 49, 49, "fp64", True),       # 2,500: 17
    ("sheet", 50, 50, "fp64", False),      # 2,601: 18 do not fit
])
def test_resident_solve_matches_separate_kernels(monkeypatch, shape, nu, nv, prec, resident):
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("row counts are those of 152 multiprocessors")
    g, rest, q = state(shape, nu, nv)
    mask = dev(S.pinned_mask(g, [0]), torch.uint8)
    rtol, tol = (1e-6, 1e-4) if prec == "mixed" else (1e-12, 1e-10)
    x, it, neg, launches = solve(monkeypatch, None, g, rest, q, prec, mask, rtol)
    x0, it0, neg0, _ = solve(monkeypatch, "host", g, rest, q, prec, mask, rtol)
    assert (launches == 1) == resident
    assert neg == neg0 == 0 and abs(it - it0) <= 1, (it, it0)
    assert np.linalg.norm(x - x0) <= tol * np.linalg.norm(x0)
    assert not x[S.pinned_mask(g, [0]).astype(bool)].any()


@pytest.mark.parametrize("prec", ["mixed", "fp64"])
def test_resident_solve_limits_curvature_and_no_mask(monkeypatch, prec):
    g, rest, q = state("sheet", 12, 9)
    for fixed in (1, 7):
        x, it, neg, _ = solve(monkeypatch, None, g, rest, q, prec, None, 1e-6, fixed=fixed)
        x0, it0, neg0, _ = solve(monkeypatch, "host", g, rest, q, prec, None, 1e-6, fixed=fixed)
        assert it == it0 == fixed and neg == neg0 == 0
        # the same few iterations: FP32 (FP64) rounding of the vectors and of the block inverses
        assert np.linalg.norm(x - x0) <= (1e-4 if prec == "mixed" else 1e-10) * np.linalg.norm(x0)
    g, rest, q = S.sheet_sinusoid(16, 3)
    _, _, neg, launches = solve(monkeypatch, None, g, rest, q, prec, None, 1e-6, mass_scale=1.0)
    _, _, neg0, _ = solve(monkeypatch, "host", g, rest, q, prec, None, 1e-6, mass_scale=1.0)
    assert neg == neg0 == 1 and launches == 1


@pytest.mark.parametrize("prec", ["mixed", "fp64"])
def test_resident_solve_wait_timeout_is_reported_and_the_shell_recovers(monkeypatch, prec):
    """With a budget of 0 polls every wait between the CTAs expires at once: the call reports
    SHELL_ERR_TIMEOUT, and with the default budget the same shell repeats its earlier solution."""
    from paper_2312_14839_gb300.bhem import Shell, ShellError
    monkeypatch.delenv("BHEM_PCG_LOOP", raising=False)
    g, rest, q = state("sheet", 12, 9)
    with Shell(g, S.SHEET_MATERIAL, dev(rest.reshape(-1)), precision=prec, assembly="color") as sh:
        _, G = sh.energy_grad_hess(dev(q.reshape(-1)), mass_scale=1e6)
        x0, it0, _ = sh.pcg_solve(-G)
        sh.set_wait_budget(0)
        with pytest.raises(ShellError) as e:
            sh.pcg_solve(-G)
        assert e.value.status == 9
        sh.set_wait_budget(-1)
        x1, it1, _ = sh.pcg_solve(-G)
        assert it1 == it0 and torch.equal(x0, x1)
