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
