"""Newton steps whose linear solves are resident, with the exchange of the solution that ends each of them (M d
and the line search's dot products formed in the same launch), against the separate kernels
(BHEM_PCG_LOOP=host), at each register form's first and last row counts; each step is repeated from the
same state, and none may run into the wait budget.

Tolerance: both forms stop at 1e-8 of the residual at the same Newton matrix, whose block-Jacobi-scaled
condition number is below 100 (M / dt^2 + K, dt = 1 ms), so displacements agree to 1e-6; atomic FP32 assembly
(the resident form of mixed precision) moves the Newton iterations by one at most."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2312_14839_gb300 import scenes as S  # noqa: E402

pytestmark = pytest.mark.gpu


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a).reshape(-1), device="cuda")


@pytest.mark.parametrize("shape,nu,nv,prec", [
    ("sheet", 10, 10, "mixed"),      # 121 nodes: 9 rows per CTA, 14 CTAs
    ("sheet", 30, 30, "mixed"),      # 961: 9 on 152 SMs
    ("annulus", 280, 5, "mixed"),    # 1,680: 12
    ("sheet", 46, 46, "mixed"),      # 2,209: 15
    ("sheet", 52, 52, "mixed"),      # 2,809: 19
    ("sheet", 64, 64, "mixed"),      # 4,225: 28
    ("sheet", 65, 65, "mixed"),      # 4,356: 29
    ("annulus", 256, 18, "mixed"),   # 4,864: 32
    ("sheet", 69, 69, "mixed"),      # 4,900: not resident
    ("sheet", 10, 10, "fp64"),       # 2
    ("sheet", 35, 37, "fp64"),       # 9
    ("sheet", 36, 36, "fp64"),       # 10
    ("sheet", 49, 49, "fp64"),       # 17
])
def test_steps_match_separate_kernels(monkeypatch, shape, nu, nv, prec):
    from paper_2312_14839_gb300 import bhem
    g, rest = S.annulus(nu, nv) if shape == "annulus" else S.flat_sheet(nu, nv, nu / max(nu, nv), nv / max(nu, nv))
    side = min(0.2 * g.dxi1 if shape == "annulus" else g.dxi1, g.dxi2)
    q0 = S.noisy(rest, 3e-3 * side, 7)
    mask = torch.as_tensor(S.pinned_mask(g, [0, g.n_nodes - 1]), device="cuda")
    params = bhem.step_params(dt=1e-3, gravity=(0.0, 0.0, -9.81), newton_max=200, pcg_max=2000)
    found = {}
    for form, repeats in ((None, 20), ("host", 1)):
        if form is None:
            monkeypatch.delenv("BHEM_PCG_LOOP", raising=False)
        else:
            monkeypatch.setenv("BHEM_PCG_LOOP", form)
        with bhem.Shell(g, S.SHEET_MATERIAL, dev(rest), precision=prec, assembly="atomic") as sh:
            states = []
            for _ in range(repeats):
                q, v = dev(q0).clone(), torch.zeros(g.n_dof, dtype=torch.float64, device="cuda")
                st = sh.newton_step(q, v, params, mask=mask, q_fixed=dev(q0))
                assert st["status"] == 0
                states.append((q.cpu().numpy(), st["newton_iters"]))
            found[form] = states
    q_ref, it_ref = found["host"][0]
    d_ref = q_ref - q0.reshape(-1)
    for q, it in found[None]:
        assert abs(it - it_ref) <= 1
        assert np.linalg.norm(q - q_ref) <= 1e-6 * np.linalg.norm(d_ref)
