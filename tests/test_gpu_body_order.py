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


@pytest.mark.parametrize("name,drop", [("quadruped", 0.38), ("biped", 0.0)])
@pytest.mark.parametrize("mode", [0, 1])
def test_environment_layer_of_a_jointed_body_0(brax, name, drop, mode):
    """Body 0 as a joint's child (it has a parent and an actuator of its own):
    observation, reward and done of each step against the oracle's formulas on
    the GPU's own states, in the one-environment kernels and in the default
    launch, with the tolerances of test_gpu_env.py."""
    from oracle import env as oenv
    d = S.SCENES[name]()
    r, order = root_last(d)
    N, T = 70, 4
    st, a = inputs(brax, d, order, N, T, drop)
    sysm = brax(r)
    if mode == 0 and sysm.paired:
        sysm.set_pair_launch(0, 1, 0)
    z = st[:, 0, 2].cpu().numpy()
    lo, hi = np.float32(np.quantile(z, 0.3)), np.float32(10.0)
    spec = dict(forward_weight=1.25, healthy_reward=0.5, ctrl_cost=0.3, min_z=float(lo), max_z=float(hi))
    for t in range(T):
        out = sysm.env_rollout(st, a[t:t + 1], auto_reset=False, **spec)
        s0, s1 = st.cpu().numpy().astype(np.float64), out["state_T"].cpu().numpy().astype(np.float64)
        obs, rew = out["obs"].cpu().numpy()[0], out["reward"].cpu().numpy()[0]
        z = s1[:, 0, 2].astype(np.float32)
        done = (z < lo) | (z > hi)
        assert np.array_equal(out["done"].cpu().numpy()[0].astype(bool), done)
        ref = oenv.observe(r, s1)
        nd = (ref.shape[1] - 11) // 2
        assert np.array_equal(obs[:, :11], ref[:, :11])
        assert np.abs(obs[:, 11:11 + nd] - ref[:, 11:11 + nd]).max() < 2e-5
        assert (np.abs(obs[:, 11 + nd:] - ref[:, 11 + nd:]) <= 1e-5 * (1.0 + np.abs(ref[:, 11 + nd:]))).all()
        ctrl = np.sum(np.clip(a[t].cpu().numpy().astype(np.float64), -1, 1) ** 2, axis=1)
        exp = 1.25 * (s1[:, 0, 0] - s0[:, 0, 0]) / r["dt"] + 0.5 * ~done - 0.3 * ctrl
        assert np.abs(rew - exp).max() < 1e-5 * (1.0 + np.abs(exp).max())
        st = out["state_T"]
    sysm.sync_status()


def test_a_cached_limb_launch_is_tuned_anew(brax, tmp_path):
    """An autotune cache that recorded the limb layout for a system whose root
    is not body 0 is not applied: the system is tuned again."""
    import json
    r, order = root_last(S.quadruped())
    sysm, cache = brax(r), str(tmp_path / "tune.json")
    st, a = inputs(brax, S.quadruped(), order, 64, 4, 0.36)
    first = sysm.autotune(st, a, cache=cache)
    table = json.load(open(cache))
    (key,) = table
    table[key].update(fwd_kernel=1, fwd_groups=1, fwd_variant=5)
    json.dump(table, open(cache, "w"))
    again = sysm.autotune(st, a, cache=cache)
    assert not first["cached"] and not again["cached"] and again["fwd_variant"] < 5
    assert sysm.autotune(st, a, cache=cache)["cached"]
