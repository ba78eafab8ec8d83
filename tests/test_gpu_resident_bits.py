"""The mixed-precision resident solve against the separate kernels, DOF by DOF: it forms every product, block
inverse and vector update with their operations in their order, so on the same matrix (colour-ordered
assembly: the same bits from run to run) it returns their solution and iteration count. Only sums over the
grid are ordered otherwise, in double-float (48 bits): a scalar of the solve rounds to another FP32
number with a chance of about 1e-5, and none may in these cases, so the bound is what FP64 outputs are
held to, 1e-9 of the norm, after a fixed number of iterations as well as at a residual of 1e-8, with the
regulariser's shift, at negative curvature and at each register form's last and first row count."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2312_14839_gb300 import scenes as S  # noqa: E402

pytestmark = pytest.mark.gpu


def dev(a, dtype=torch.float64):
    return torch.as_tensor(np.ascontiguousarray(a).reshape(-1), dtype=dtype, device="cuda")


def solves(monkeypatch, form, g, rest, q, mask, calls, mass_scale):
    from paper_2312_14839_gb300.bhem import Shell
    if form is None:
        monkeypatch.delenv("BHEM_PCG_LOOP", raising=False)
    else:
        monkeypatch.setenv("BHEM_PCG_LOOP", form)
    with Shell(g, S.SHEET_MATERIAL, dev(rest), precision="mixed", assembly="color") as sh:
        _, G = sh.energy_grad_hess(dev(q), mass_scale=mass_scale)
        out = []
        for kw in calls:
            n0 = sh.kernel_launches()
            x, it, neg = sh.pcg_solve(-G, mask=mask, max_iter=2000, **kw)
            out.append((x.cpu().numpy(), it, neg, sh.kernel_launches() - n0))
        return out


def assert_same(a, b):
    for (x, it, neg, launches), (x0, it0, neg0, _) in zip(a, b):
        assert launches == 1 and (it, neg) == (it0, neg0)
        assert np.linalg.norm(x - x0) <= 1e-9 * np.linalg.norm(x0)


@pytest.mark.parametrize("shape,nu,nv", [
    ("sheet", 1, 1), ("annulus", 2, 1), ("annulus", 7, 2), ("sheet", 12, 9),
    ("sheet", 30, 30),       # 961 nodes: 9 rows per CTA on 152 SMs
    ("annulus", 280, 5),     # 1,680: 12
    ("sheet", 44, 44),       # 2,025: 14, one pass of the matrix in registers
    ("sheet", 46, 46),       # 2,209: 15, two
    ("sheet", 64, 64),       # 4,225: 28
    ("sheet", 65, 65),       # 4,356: 29, from shared memory
    ("annulus", 256, 18),    # 4,864: 32
])
def test_resident_solve_has_the_separate_kernels_solution(monkeypatch, shape, nu, nv):
    if shape == "annulus":
        g, rest = S.annulus(nu, nv)
        side = min(0.2 * g.dxi1, g.dxi2)
    else:
        g, rest = S.flat_sheet(nu, nv, nu / max(nu, nv), nv / max(nu, nv))
        side = min(g.dxi1, g.dxi2)
    q = S.noisy(rest, 3e-3 * side, 5)
    mask = dev(S.pinned_mask(g, [0]), torch.uint8)
    calls = [dict(rtol=1e-8), dict(fixed_iters=1), dict(fixed_iters=50), dict(rtol=1e-8, tau=0.1)]
    assert_same(solves(monkeypatch, None, g, rest, q, mask, calls, 1e6),
                solves(monkeypatch, "host", g, rest, q, mask, calls, 1e6))


def test_resident_solve_of_an_indefinite_matrix_has_the_separate_kernels_solution(monkeypatch):
    g, rest, q = S.sheet_sinusoid(24, 3)   # indefinite without the shift, and slow to converge with it
    calls = [dict(rtol=1e-6), dict(fixed_iters=50, tau=1.0), dict(fixed_iters=200, tau=10.0)]
    a = solves(monkeypatch, None, g, rest, q, None, calls, 1.0)
    assert a[0][2] == 1
    assert_same(a, solves(monkeypatch, "host", g, rest, q, None, calls, 1.0))
