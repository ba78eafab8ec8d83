"""Dispatch of the mixed-precision resident solve at the number of rows whose DOFs a CTA's threads own, 32: the
largest shells it takes and the first ones beyond (33 and 34 rows per CTA on 152 SMs), which fit the
shared memory but go to the separate kernels. Against the separate kernels, as in
test_gpu_resident.py: iteration counts within one and solutions to 1e-4 at a residual of 1e-6."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2312_14839_gb300 import scenes as S  # noqa: E402

pytestmark = pytest.mark.gpu


def dev(a, dtype=torch.float64):
    return torch.as_tensor(np.ascontiguousarray(a).reshape(-1), dtype=dtype, device="cuda")


@pytest.mark.parametrize("assembly", ["color", "atomic"])
@pytest.mark.parametrize("shape,nu,nv,resident", [
    ("sheet", 67, 70, True),        # 4,828 nodes: 32 rows, the last CTA short
    ("annulus", 256, 18, True),     # 4,864: 32 in all of 152 CTAs
    ("annulus", 35, 138, False),    # 4,865: 33, one row in the last CTA
    ("sheet", 69, 69, False),       # 4,900: 33
    ("annulus", 280, 17, False),    # 5,040: 34
    ("sheet", 70, 70, False),       # 5,041: 34
])
def test_every_accepted_row_is_solved(monkeypatch, shape, nu, nv, resident, assembly):
    from paper_2312_14839_gb300.bhem import Shell
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("row counts are those of 152 multiprocessors")
    g, rest = S.annulus(nu, nv) if shape == "annulus" else S.flat_sheet(nu, nv, nu / max(nu, nv), nv / max(nu, nv))
    side = min(0.2 * g.dxi1 if shape == "annulus" else g.dxi1, g.dxi2)
    q = S.noisy(rest, 3e-3 * side, 5)
    mask = dev(S.pinned_mask(g, [0]), torch.uint8)
    found = {}
    for form in (None, "host"):
        if form is None:
            monkeypatch.delenv("BHEM_PCG_LOOP", raising=False)
        else:
            monkeypatch.setenv("BHEM_PCG_LOOP", form)
        with Shell(g, S.SHEET_MATERIAL, dev(rest), precision="mixed", assembly=assembly) as sh:
            _, G = sh.energy_grad_hess(dev(q), mass_scale=1e6)
            n0 = sh.kernel_launches()
            x, it, neg = sh.pcg_solve(-G, mask=mask, rtol=1e-6, max_iter=2000)
            found[form] = x.cpu().numpy(), it, neg, sh.kernel_launches() - n0
    x, it, neg, launches = found[None]
    x0, it0, neg0, _ = found["host"]
    assert (launches == 1) == resident
    assert neg == neg0 == 0 and abs(it - it0) <= 1
    assert np.linalg.norm(x - x0) <= 1e-4 * np.linalg.norm(x0)
