"""Systems whose tree's root is not body 0: the torso path and the environment
layer follow body 0, whatever its place in the tree, in the default launch as
in every other kernel."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2106_13281_gb300 import scenes as S

pytestmark = pytest.mark.gpu

PER_BODY = ("mass", "inertia", "rest_pos", "rest_rot", "frozen_pos", "frozen_rot")


@pytest.fixture(scope="module")
def brax():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2106_13281_gb300.system import BraxSystem
    return BraxSystem


def root_last(d):
    """The same system with its bodies renumbered, body 0 last; and the old index of each body."""
    B = len(d["mass"])
    order = np.roll(np.arange(B), -1)
    new = np.argsort(order)
    r = dict(d)
    for k in PER_BODY:
        r[k] = np.asarray(d[k])[order]
    for k in ("parent", "child"):
        r[k] = new[d[k]].astype(np.int32)
    r["col_body"] = np.where(d["col_body"] < 0, -1, new[d["col_body"]]).astype(np.int32)
    r["body_names"] = [d["body_names"][i] for i in order]
    return r, order


def inputs(brax, d, order, N, T, drop):
    rp, rr, ang = S.initial_conditions(d, N, 41, height_jitter=0.05)
    rp[:, 2] -= drop
    f32 = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()
    st = brax(d).default_qp(N, f32(rp), f32(rr), f32(ang))[:, torch.from_numpy(order).cuda()].contiguous()
    return st, f32(S.actions(d, N, T, 42))


@pytest.mark.parametrize("name,drop", [("quadruped", 0.36), ("pendulum", 0.0)])
@pytest.mark.parametrize("N", [1, 70, 20000])
def test_torso_and_environment_follow_body_0(brax, name, drop, N):
    """The default launch against the paired body-layout kernel: the same bits
    in every output, and the torso path's last step is body 0's position."""
    d = S.SCENES[name]()
    r, order = root_last(d)
    T = 5
    st, a = inputs(brax, d, order, N, T, drop)
    default, paired = brax(r), brax(r)
    paired.set_pair_launch(1, 1, 1)
    z = st[:, 0, 2].float()
    spec = dict(min_z=float(z.quantile(0.3)) if N > 1 else 0.0, max_z=10.0)
    got = default.rollout(st, a, K=2, checkpoints=True, torso=True, contact_count=True)
    ref = paired.rollout(st, a, K=2, checkpoints=True, torso=True, contact_count=True)
    assert torch.equal(ref["torso"][-1], ref["state_T"][:, 0, :3])
    for k in ref:
        assert torch.equal(got[k], ref[k]), k
    got, ref = default.env_rollout(st, a, **spec), paired.env_rollout(st, a, **spec)
    for k in ref:
        assert torch.equal(got[k], ref[k]), k
    default.sync_status()
