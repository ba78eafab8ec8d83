"""Rays and moving points aimed at nodes and at the middle of patch edges, where candidates of several patches
have equal keys, and points that start on the surface: the searches without statistics, which leave
sub-patches out, return bit for bit what the searches with statistics return, the patch among them."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2312_14839_gb300 import scenes as S  # noqa: E402

pytestmark = pytest.mark.gpu


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


def on_edges(g, p):
    """Nodes and midpoints (of the nodes' positions) of the grid lines that are not seams."""
    i = np.arange(len(p))
    a, b = i[i % g.n1 < g.n1 - 1], i[i < len(p) - g.n1]
    return np.concatenate([p, 0.5 * (p[a] + p[a + 1]), 0.5 * (p[b] + p[b + g.n1])])


def same(full, culled, least):
    for k in culled:
        np.testing.assert_array_equal(culled[k].cpu().numpy(), full[k].cpu().numpy(), err_msg=k)
    assert int((culled["flags"] & 1).sum()) > least


@pytest.mark.parametrize("variant", ["newton", "midpoint"])
@pytest.mark.parametrize("name", ["plane", "cylinder", "drape"])
def test_rays(name, variant):
    from paper_2312_14839_gb300.bhem import Shell
    g, q, eye, _ = S.ray_scenes()[name]
    t = on_edges(g, q[:, :3])[::3]
    o, d = [], []
    for e in (np.array(eye), np.array(eye) * [1.0, -1.0, 1.0], np.array([0.5, 0.5, 3.0]), np.array([0.0, 0.0, 0.5])):
        n = np.linalg.norm(t - e, axis=1)
        far = n > 1e-6
        o.append(np.tile(e, (far.sum(), 1)))
        d.append((t - e)[far] / n[far, None])
    for u in np.array([[1, 0, 0], [0, 1, 0], [0, 0, 1], [1, 1, 0], [1, 0, 1], [1, 1, 1], [0, 1, -1], [1, -1, 0]]):
        for sign in (1.0, -1.0):
            u1 = sign * u / np.linalg.norm(u)
            o.append(t - 2.0 * u1)
            d.append(np.tile(u1, (len(t), 1)))
    o, d = dev(np.concatenate(o)), dev(np.concatenate(d))
    with Shell(g, S.SHEET_MATERIAL, dev(q).reshape(-1), precision="mixed") as sh:
        dq = dev(q).reshape(-1)
        same(sh.trace_rays(dq, o, d, variant=variant, want_stats=True), sh.trace_rays(dq, o, d, variant=variant), 1000)


@pytest.mark.parametrize("variant", ["newton", "midpoint"])
@pytest.mark.parametrize("moving", [True, False])
@pytest.mark.parametrize("name", ["plane", "cylinder", "drape"])
def test_points(name, moving, variant):
    from paper_2312_14839_gb300.bhem import Shell
    g, q, dq, _, _ = S.ccd_scene(name, 100, 3)
    dq = dq if moving else 0.0 * dq
    a, b = on_edges(g, q[:, :3])[::2], on_edges(g, (q + dq)[:, :3])[::2]
    x0, dx = [], []
    # the last: on the surface; not along the cylinder's wall, where a search takes seconds
    offsets = ([0, 0, 0.5], [0, 0, -0.25], [0.5, 0, 0], [0.25, 0.25, 0.25], [0, 0, 0])
    for off in offsets[2:] if name == "cylinder" else offsets:
        for s in (0.25, 0.5, 0.75):   # meets the surface about then
            x0.append(a + np.array(off, dtype=float))
            dx.append((a + s * (b - a) - x0[-1]) / s)
        x0.append(x0[-1])
        dx.append(np.tile(-2.0 * np.array(off, dtype=float), (len(a), 1)))
    args = [dev(q).reshape(-1), dev(dq).reshape(-1), dev(np.concatenate(x0)), dev(np.concatenate(dx))]
    with Shell(g, S.SHEET_MATERIAL, dev(q).reshape(-1), precision="mixed") as sh:
        same(sh.ccd_points(*args, variant=variant, want_stats=True), sh.ccd_points(*args, variant=variant), 800)
