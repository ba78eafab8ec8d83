"""Ray directions of any length: tau counts in units of d, and the search without statistics, which leaves out
sub-patches beyond the best hit by their distance along the ray, returns bit for bit the hits of the search
with statistics, which leaves out none. Camera rays, rays that meet the cylinder twice and the drape several
times, directions from 1e-8 to 1e20 long and single components that FP32 cannot hold; a zero direction."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2312_14839_gb300 import scenes as S  # noqa: E402

pytestmark = pytest.mark.gpu


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


def rays(name):
    g, q, eye, tgt = S.ray_scenes()[name]
    o, d = S.camera_rays(60, 45, eye, tgt)
    rng = np.random.default_rng(5)
    lo, hi = q[:, :3].min(0) - 0.05, q[:, :3].max(0) + 0.05
    a, b = rng.uniform(lo, hi, size=(1500, 3)), rng.uniform(lo, hi, size=(1500, 3))
    # along the sheet: several crossings of a drape, in and out of a cylinder
    b[:750, 2] = a[:750, 2]
    u = (b - a) / np.linalg.norm(b - a, axis=1, keepdims=True)
    return g, q, np.concatenate([o, a - 0.5 * u]), np.concatenate([d, u])


@pytest.mark.parametrize("variant", ["newton", "midpoint"])
@pytest.mark.parametrize("name", ["plane", "cylinder", "drape"])
def test_culled_search_gives_the_same_hits(name, variant):
    from paper_2312_14839_gb300.bhem import Shell
    g, q, o, d = rays(name)
    with Shell(g, S.SHEET_MATERIAL, dev(q).reshape(-1), precision="mixed") as sh:
        dq, do = dev(q).reshape(-1), dev(o)
        first = None
        for scale in (1.0, 3.0, 0.2, 100.0, 1e-3, 1e-8, 1e8, 1e20):
            dd = dev(d * scale)
            full = sh.trace_rays(dq, do, dd, variant=variant, want_stats=True)
            culled = sh.trace_rays(dq, do, dd, variant=variant)
            for k in culled:
                np.testing.assert_array_equal(culled[k].cpu().numpy(), full[k].cpu().numpy(), err_msg=f"{scale} {k}")
            hit = (culled["flags"] & 1).bool().cpu()
            if first is None:
                first = hit
                assert 300 < int(hit.sum()) < len(o)
            if 1e-3 <= scale <= 100.0:   # the same rays (but for those that touch an edge)
                assert int((hit != first).sum()) <= 0.01 * len(o)
        odd = d.copy()   # components out of FP32's range beside ordinary ones, and no direction at all
        odd[::3, 0] = 1e-35
        odd[1::3, 1] = 1e-42
        odd[2::3, 2] = 1e35
        odd[::50] = 0.0
        dd = dev(odd)
        full = sh.trace_rays(dq, do, dd, variant=variant, want_stats=True)
        culled = sh.trace_rays(dq, do, dd, variant=variant)
        for k in culled:
            np.testing.assert_array_equal(culled[k].cpu().numpy(), full[k].cpu().numpy(), err_msg=k)
