"""A batch step's rounding: strips one patch wide, whose sums over patches have one value in any order, two Newton
iterations of 12 PCG iterations each, against states recorded before the batch's kernels were rearranged
(tests/golden/batch_strips.json, FP64 as hexadecimal). The FP32 products and vector updates keep their operations and
their order, so the states agree to what FP64 sums in another order leave, 1e-9 of the displacement; with the
products of a row chained otherwise such strips came out up to 2e-5 apart."""
import json
import os

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2312_14839_gb300 import scenes as S  # noqa: E402

GOLDEN = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "batch_strips.json")
PATCHES = (17, 40, 9, 31)


def strips():
    return [S.flat_sheet(n, 1, 1.0, 1.0 / n) for n in PATCHES]


def step(assembly):
    """(initial state, state after the step, velocities)."""
    from paper_2312_14839_gb300 import bhem
    sheets = strips()
    mats = [m for _, m, _, _ in S.batch_sheets(len(sheets), seed=4)]
    q0 = np.concatenate([S.noisy(rest, 3e-5, [1, k]).reshape(-1) for k, (_, rest) in enumerate(sheets)])
    mask = np.concatenate([S.pinned_mask(g, [0, g.n_nodes - 1]) for g, _ in sheets])
    dev = lambda a: torch.as_tensor(a, device="cuda")   # noqa: E731
    with bhem.Batch([(g, m, rest) for (g, rest), m in zip(sheets, mats)], stream=torch.cuda.current_stream(),
                    assembly=assembly) as b:
        q, v = dev(q0).clone(), torch.zeros(len(q0), dtype=torch.float64, device="cuda")
        b.newton_step(q, v, bhem.step_params(dt=1e-3, newton_max=2, pcg_fixed_iters=12), mask=dev(mask), q_fixed=dev(q0))
        torch.cuda.synchronize()
        return q0, q.cpu().numpy(), v.cpu().numpy()


@pytest.mark.gpu
@pytest.mark.parametrize("assembly", ["atomic", "color"])
def test_states_are_the_recorded_ones(assembly):
    with open(GOLDEN) as f:
        golden = json.load(f)
    q0, q, v = step(assembly)
    at = np.array(golden["dofs"])
    d = np.array([float.fromhex(x) for x in golden["displacement"]])
    assert np.linalg.norm((q - q0)[at] - d) <= 1e-9 * np.linalg.norm(d)
    w = np.array([float.fromhex(x) for x in golden["velocity"]])
    assert np.linalg.norm(v[at] - w) <= 1e-9 * np.linalg.norm(w)
