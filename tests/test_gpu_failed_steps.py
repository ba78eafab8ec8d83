"""A step that ends in an error other than SHELL_ERR_NOT_CONVERGED leaves q and v as they were, wherever it
fails: with a wait budget of 0 polls (in the first element pass of mixed precision, in the linear solve of
FP64, which is resident) and at a prescribed position that collapses a patch, on device and on host arrays,
with prescribed DOFs and a warm start that have replaced q by then."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2312_14839_gb300 import scenes as S  # noqa: E402

pytestmark = pytest.mark.gpu

DEGENERATE, TIMEOUT = 4, 9


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a).reshape(-1), device="cuda")


@pytest.mark.parametrize("where", ["device", "host"])
@pytest.mark.parametrize("warm", [False, True])
@pytest.mark.parametrize("prec", ["mixed", "fp64"])
@pytest.mark.parametrize("cause", ["budget", "collapse"])
def test_q_and_v_are_unchanged(monkeypatch, cause, prec, warm, where):
    from paper_2312_14839_gb300 import bhem
    monkeypatch.delenv("BHEM_PCG_LOOP", raising=False)
    g, rest = S.flat_sheet(12, 9, 1.0, 0.75)
    q0 = S.noisy(rest, 1e-3, 3).reshape(-1)
    v0 = np.random.Generator(np.random.PCG64(4)).standard_normal(g.n_dof) * 1e-2
    mask = S.pinned_mask(g, range(g.n_nodes) if cause == "collapse" else [0], kinds=(0, 1, 2, 3))
    target = np.zeros(g.n_dof) if cause == "collapse" else q0 + 1e-3
    put = dev if where == "device" else (lambda a: np.array(a, dtype=a.dtype))
    params = bhem.step_params(dt=1e-3, gravity=(0.0, 0.0, -9.81))
    with bhem.Shell(g, S.SHEET_MATERIAL, dev(rest), precision=prec) as sh:
        q, v = put(q0), put(v0)
        kw = dict(mask=put(mask), q_fixed=put(target), warm=put(q0 + 2e-4) if warm else None)
        if cause == "budget":
            sh.set_wait_budget(0)
        with pytest.raises(bhem.ShellError) as e:
            sh.newton_step(q, v, params, **kw)
        assert e.value.status == (TIMEOUT if cause == "budget" else DEGENERATE)
        same = (lambda a, b: torch.equal(a, dev(b))) if where == "device" else np.array_equal
        assert same(q, q0) and same(v, v0)
        if cause == "budget":   # and the shell goes on
            sh.set_wait_budget(-1)
            assert sh.newton_step(q, v, params, **kw)["status"] == 0
            assert not same(q, q0)
