"""A patch's results do not depend on the form that its grid's size selects. On a strip of one patch across
every node has at most two patches, so sums over patches have one value whatever their order, and a long
strip that begins with a short one's nodes has to repeat its results bit for bit away from the short
one's end."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2312_14839_gb300 import scenes as S  # noqa: E402

pytestmark = pytest.mark.gpu

SHORT, LONG = 300, 2400   # patches: a warp each / half a warp each, on 152 SMs; one per warp of a launch / several


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a).reshape(-1), device="cuda")


def strips(noise, seed):
    """The same first SHORT + 1 columns of nodes on both grids: (grid, rest, q) of each."""
    out = []
    rng = np.random.Generator(np.random.PCG64(seed))
    d = None
    for n in (LONG, SHORT):
        g, rest = S.flat_sheet(n, 1, float(n) / SHORT, 1.0 / SHORT)
        if d is None:
            d = noise * rng.standard_normal((2, LONG + 1, 12))
        out.append((g, rest, rest + d[:, : n + 1].reshape(-1, 12)))
    return out


def columns(a):
    return a.reshape(2, -1, 12)[:, :SHORT]


@pytest.mark.parametrize("noise", [1e-6, 3e-5])
def test_gradient_of_a_patch_is_the_same_by_a_warp_and_by_half_a_warp(noise):
    from paper_2312_14839_gb300.bhem import Shell
    G = []
    for g, rest, q in strips(noise, 1):
        with Shell(g, S.SHEET_MATERIAL, dev(rest), precision="mixed") as sh:
            G.append(sh.energy_grad_hess(dev(q), want_hessian=False)[1].cpu().numpy())
    a, b = map(columns, G)
    assert np.array_equal(a, b)


@pytest.mark.parametrize("n", [1, 7, SHORT, LONG])
@pytest.mark.parametrize("fixed", [10, 0])
def test_steps_of_a_strip_do_not_depend_on_the_assembly(n, fixed):
    """Colour-ordered and atomic assembly of a strip form the same sums, so a step has the same Hessians; its
    linear solves are the separate kernels' and the resident one, whose solutions agree (1e-9, as in
    test_gpu_resident_bits.py)."""
    from paper_2312_14839_gb300 import bhem
    g, rest = S.flat_sheet(n, 1, float(n) / SHORT, 1.0 / SHORT)
    q0 = S.noisy(rest, 3e-5, 2)
    mask = dev(S.pinned_mask(g, [0, g.n_nodes - 1]))
    params = bhem.step_params(dt=1e-3, gravity=(0.0, 0.0, -9.81), newton_max=2 if fixed else 200, pcg_max=2000,
                              pcg_fixed_iters=fixed)
    out = []
    for assembly in ("color", "atomic"):
        with bhem.Shell(g, S.SHEET_MATERIAL, dev(rest), precision="mixed", assembly=assembly) as sh:
            q, v = dev(q0).clone(), torch.zeros(g.n_dof, dtype=torch.float64, device="cuda")
            st = sh.newton_step(q, v, params, mask=mask, q_fixed=dev(q0))
            out.append((q.cpu().numpy(), v.cpu().numpy(), st["newton_iters"], st["status"]))
    (qa, va, ia, sa), (qb, vb, ib, sb) = out
    assert (ia, sa) == (ib, sb)
    assert np.linalg.norm(qa - qb) <= 1e-9 * np.linalg.norm(qa) and np.linalg.norm(va - vb) <= 1e-9 * np.linalg.norm(va)
