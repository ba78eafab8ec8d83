"""Which calls of shell_energy_grad_hess evaluate energy, gradient and Hessian in one pass over the elements: on
152 SMs atomic assembly with up to 1,824 patches (one per warp) or 3,648 and more (two). The others take
the energy kernel, so their energy is bit for bit the one of a call without the Hessian. In one pass
the patches' energies are the same numbers summed in another order: np additions of rounding 2^-53."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2312_14839_gb300 import scenes as S  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("assembly,nu,nv,one_pass", [
    ("color", 6, 6, False), ("color", 40, 40, False), ("color", 64, 64, False),
    ("atomic", 1, 1, True), ("atomic", 48, 38, True),      # 1,824
    ("atomic", 365, 5, False), ("atomic", 45, 45, False), ("atomic", 3647, 1, False),
    ("atomic", 64, 57, True), ("atomic", 64, 64, True),    # 3,648
])
def test_energy_with_and_without_the_hessian(assembly, nu, nv, one_pass):
    from paper_2312_14839_gb300.bhem import Shell
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("patch counts are those of 152 multiprocessors")
    g, rest = S.flat_sheet(nu, nv, nu / max(nu, nv), nv / max(nu, nv))
    q = S.noisy(rest, 1e-2 * g.dxi1, 3)
    d = lambda a: torch.as_tensor(np.ascontiguousarray(a).reshape(-1), device="cuda")   # noqa: E731
    with Shell(g, S.SHEET_MATERIAL, d(rest), precision="mixed", assembly=assembly) as sh:
        E, G = sh.energy_grad_hess(d(q), mass_scale=1e6)
        V = sh.bsr()[2]
        E0, G0 = sh.energy_grad_hess(d(q), want_hessian=False)
        sh.energy_grad_hess(d(q), mass_scale=1e6, want_energy=False, want_grad=False)
        V0 = sh.bsr()[2]
    if one_pass:
        assert abs(E.item() - E0.item()) <= g.n_patches * 2.0**-53 * E0.item()
    else:
        assert E.item() == E0.item()
    # at most four patches per node, in FP64 and FP32 atomics of any order; FP32 roundings may differ in one pass
    assert torch.linalg.norm(G - G0) <= 4 * 2.0**-53 * torch.linalg.norm(G0) * 4
    assert torch.linalg.norm(V - V0) <= 1e-6 * torch.linalg.norm(V0)
