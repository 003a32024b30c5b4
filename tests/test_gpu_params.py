"""General systems whose launch keeps only the pairs' parameters in shared
memory (or none, without pairs): one step and the adjoint of one substep against
the FP64 oracle, with the tolerances of test_gpu_general.py and
test_gpu_adjoint.py.  The sizes: the pairs' at any number of environments (9
bodies and 10 pairs forward, 5 and 10 both ways), below one block an SM (10 and
20, reverse), above it (12 and 45, forward; no pairs: the pool)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import oracle as orc
from paper_2106_13281_gb300 import scenes as S
from parity_util import decided_envs
from test_gpu_general import cloud

pytestmark = pytest.mark.gpu

CASES = [(9, 10, 70), (5, 10, 70), (10, 20, 70), (12, 45, 32 * 153 + 1), (0, 0, 32 * 153 + 1)]


def setup(bodies, pairs, N, substeps):
    d = cloud(bodies, pairs) if bodies else S.SCENES["quadruped_2dof"]()
    d = dict(d, dt=float(d["dt"]) / int(d["substeps"]) * substeps, substeps=substeps)
    rng = np.random.default_rng(17)
    st = np.zeros((N, len(d["mass"]), 13))
    st[..., 0:3], st[..., 3:7] = d["rest_pos"], d["rest_rot"]
    if bodies:  # the free bodies of the heap move against each other
        st[..., 0:3] += 0.02 * rng.normal(size=st[..., 0:3].shape)
        st[..., 3:7] += 0.05 * rng.normal(size=st[..., 3:7].shape)
        st[..., 3:7] /= np.linalg.norm(st[..., 3:7], axis=-1, keepdims=True)
    st[..., 7:13] = 0.3 * rng.normal(size=st[..., 7:13].shape)
    st = st.astype(np.float32).astype(np.float64)
    return d, st, S.actions(d, N, 1, 18).astype(np.float64), rng


cu = lambda x: torch.from_numpy(np.ascontiguousarray(x, dtype=np.float32)).cuda()


@pytest.mark.parametrize("bodies,pairs,N", CASES)
def test_one_step_parity(bodies, pairs, N):
    from paper_2106_13281_gb300.system import BraxSystem
    d, st, a, _ = setup(bodies, pairs, N, 2)
    sysm = BraxSystem(d)
    ref, count = orc.rollout(d, st, a, contact_count=True)
    out = sysm.rollout(cu(st), cu(a), contact_count=True)
    sysm.sync_status()
    ok = decided_envs(d, st, a)
    assert ok.mean() >= 0.5 and (not bodies or count.sum() > 0)
    err = np.abs(out["state_T"].cpu().numpy() - ref)[ok]
    assert err[..., 0:3].max() <= 1e-5 and err[..., 3:7].max() <= 1e-4
    assert err[..., 7:10].max() <= 2e-4 and err[..., 10:13].max() <= 4e-3
    assert np.mean(out["contact_count"].cpu().numpy()[ok] == count[ok]) >= 0.9


@pytest.mark.parametrize("bodies,pairs,N", CASES[:3])
def test_single_substep_adjoint(bodies, pairs, N):
    from paper_2106_13281_gb300.system import BraxSystem
    d, st, a, rng = setup(bodies, pairs, N, 1)
    sysm = BraxSystem(d)
    g = rng.normal(size=st.shape).astype(np.float32).astype(np.float64)
    out = sysm.rollout(cu(st), cu(a), K=1, checkpoints=True, contact_count=True)
    _, gs = sysm.rollout_backward(cu(st), cu(a), out["checkpoints"], cu(g), K=1)
    sysm.sync_status()
    _, gs_ref = orc.vjp(d, st, a, g)
    _, count = orc.rollout(d, st, a, contact_count=True)
    ok = decided_envs(d, st, a) & (out["contact_count"].cpu().numpy() == count)
    assert ok.mean() >= 0.5 and count[ok].sum() > 0
    gs = gs.cpu().numpy().astype(np.float64)
    rel = [np.linalg.norm(gs[n] - gs_ref[n]) / np.linalg.norm(gs_ref[n]) for n in range(N) if ok[n]]
    assert max(rel) < 1e-3
