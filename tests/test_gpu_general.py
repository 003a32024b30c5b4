"""The general kernel's branches that no scene of scenes.py reaches, one step
against the FP64 oracle from identical states (the tolerances of
test_gpu_forward.py): a system whose parameters do not fit shared memory beside
its groups (they come from the constant pool), bodies with several pair
colliders (their geometry is not published; the broadphase tests them in the
narrow phase), and fewer pairs than warps."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import oracle as orc
from paper_2106_13281_gb300 import scenes as S
from parity_util import decided_envs

pytestmark = pytest.mark.gpu


def cloud(n, most):
    """n free capsules in a loose heap, their first `most` pairs tested."""
    sb = S.SceneBuilder(dt=0.01, substeps=2)
    rng = np.random.default_rng(5)
    for i in range(n):
        axis = rng.normal(size=3)
        sb.capsule_body(f"c{i}", 1.0, 0.06, 0.3, rng.uniform(-0.35, 0.35, 3) + (0, 0, 0.6), axis, inertia=(0.1, 0.1, 0.1))
    for a in range(n):
        for b in range(a + 1, n):
            if len(sb.pairs) < most:
                sb.pair(sb.collider_of(a), sb.collider_of(b))
    return sb.build()


def dumbbells():
    """Two bodies of four capsules each, every capsule against every other: 16
    pairs for two warps, no body with a single pair collider."""
    sb = S.SceneBuilder(dt=0.01, substeps=2)
    cols = []
    for k, z in enumerate((0.5, 0.72)):
        b = sb.body(f"d{k}", 1.0, (0.1, 0.12, 0.15), (0.02 * k, 0, z))
        cols.append([sb.collider(b, S.CAPSULE, pos=(0.16 * i - 0.24, 0, 0), radius=0.1, length=0.3) for i in range(4)])
    ground = sb.plane()
    for a in cols[0]:
        sb.pair(a, ground)
        for b in cols[1]:
            sb.pair(a, b)
    return sb.build()


@pytest.mark.parametrize("name", ["cloud18", "cloud3", "dumbbells"])
@pytest.mark.parametrize("N", [1, 33])
def test_one_step_parity(name, N):
    from paper_2106_13281_gb300.system import BraxSystem
    d = {"cloud18": lambda: cloud(18, 127), "cloud3": lambda: cloud(3, 3), "dumbbells": dumbbells}[name]()
    sysm = BraxSystem(d)
    rng = np.random.default_rng(11)
    B = len(d["mass"])
    st = np.zeros((N, B, 13))
    st[..., 0:3] = d["rest_pos"] + 0.02 * rng.normal(size=(N, B, 3))
    st[..., 3:7] = d["rest_rot"] + 0.05 * rng.normal(size=(N, B, 4))
    st[..., 3:7] /= np.linalg.norm(st[..., 3:7], axis=-1, keepdims=True)
    st[..., 7:13] = 0.3 * rng.normal(size=(N, B, 6))
    st = st.astype(np.float32).astype(np.float64)
    a = np.zeros((1, N, 0))
    ref, count = orc.rollout(d, st, a, contact_count=True)
    cu = lambda x: torch.from_numpy(np.ascontiguousarray(x, dtype=np.float32)).cuda()
    out = sysm.rollout(cu(st), cu(a), contact_count=True)
    sysm.sync_status()
    got = out["state_T"].cpu().numpy()
    ok = decided_envs(d, st, a)
    assert ok.mean() >= 0.5 and (name == "cloud3" or count.sum() > 0)
    err = np.abs(got - ref)[ok]
    assert err[..., 0:3].max() <= 1e-5 and err[..., 3:7].max() <= 1e-4
    assert err[..., 7:10].max() <= 2e-4 and err[..., 10:13].max() <= 4e-3
    assert np.mean(out["contact_count"].cpu().numpy()[ok] == count[ok]) >= 0.9
