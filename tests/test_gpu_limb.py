"""The limb-layout kernels (one root, L limbs of two hinged bodies): the wide
kernel (a limb of two environments a lane) and the split kernel (a limb body a
lane) against the paired body-layout kernel, which computes the same operations
in the same order: every output equal, at the edges of a warp's and a block's
environments, for every supported number of limbs, with frozen axes, anisotropic
inertias, the environment layer and the chunked schedule."""
import numpy as np
import pytest
import torch

from paper_2106_13281_gb300 import scenes as S

pytestmark = pytest.mark.gpu

WIDE, SPLIT = 6, 7


@pytest.fixture(scope="module")
def brax():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2106_13281_gb300.system import BraxSystem
    return BraxSystem


def crawler(limbs):
    """A torso with `limbs` legs of two capsules each around it."""
    sb = S.SceneBuilder()
    t = sb.body("torso", 10.0, S.UNIT_INERTIA, (0, 0, 0.75))
    sb.collider(t, S.CAPSULE, radius=0.25, length=0.5)
    ground = sb.plane()
    sb.pair(sb.collider_of(t), ground)
    ez = np.array([0.0, 0, 1])
    for k in range(limbs):
        phi = 0.3 + 2 * np.pi * k / limbs
        d = np.array([np.cos(phi), np.sin(phi), 0.0])
        hip = np.array([0, 0, 0.75]) + 0.25 * d
        knee = hip + 0.4 * d
        th = sb.capsule_body(f"thigh{k}", 1.0, 0.08, 0.4, hip + 0.2 * d, d, inertia=S.UNIT_INERTIA)
        sh = sb.capsule_body(f"shin{k}", 1.0, 0.08, 0.4, knee + 0.2 * d, d, inertia=S.UNIT_INERTIA)
        jh = sb.joint(t, th, hip, axis=ez, ref=d, limits=((-30, 30),), **S.QUADRUPED_JOINT)
        jk = sb.joint(th, sh, knee, axis=np.cross(ez, d), ref=d, limits=((30, 70),), **S.QUADRUPED_JOINT)
        sb.actuator(jh, 0, 150.0)
        if limbs != 2:  # two limbs: hips only, so that the lower bodies have no actuator
            sb.actuator(jk, 0, 150.0)
        sb.pair(sb.collider_of(th), ground)
        sb.pair(sb.collider_of(sh), ground)
    return sb.build()


SCENES = {"quadruped": S.quadruped, "pendulum": S.pendulum, "planar": lambda: S.planar(S.quadruped()),
          "aniso": S.quadruped_aniso, "crawler2": lambda: crawler(2), "crawler8": lambda: crawler(8)}


def inputs(sysm, d, N, T):
    rp, rr, ang = S.initial_conditions(d, N, 31, height_jitter=0.05)
    if len(d["parent"]) > 2:
        rp[:, 2] -= 0.36  # on the ground
    f32 = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()
    return sysm.default_qp(N, f32(rp), f32(rr), f32(ang)), f32(S.actions(d, N, T, 32))


def same(a, b):
    for k in b:
        assert torch.equal(a[k], b[k]), k


@pytest.mark.parametrize("name", list(SCENES))
@pytest.mark.parametrize("N", [1, 3, 16, 65, 1027])
def test_limb_kernels_equal_the_paired_kernel(brax, name, N):
    d = SCENES[name]()
    sysm = brax(d)
    T = 12
    st, a = inputs(sysm, d, N, T)
    sysm.set_pair_launch(1, 1, 1)
    ref = sysm.rollout(st, a, K=5, checkpoints=True, torso=True, contact_count=True)
    env = sysm.env_rollout(st, a, min_z=0.3, max_z=0.8)
    sysm.sync_status()
    for v in (WIDE, SPLIT):
        sysm.set_pair_launch(1, 1, v)
        same(sysm.rollout(st, a, K=5, checkpoints=True, torso=True, contact_count=True), ref)
        same(sysm.env_rollout(st, a, min_z=0.3, max_z=0.8), env)
        sysm.set_schedule(2, 5)
        same(sysm.rollout(st, a, K=5, checkpoints=True, torso=True, contact_count=True), ref)
        sysm.set_schedule(1)
        sysm.sync_status()


def test_default_launch_is_the_limb_layout_on_both_sides_of_its_rule(brax):
    """The default launch (no launch override) at a size of each kernel and a
    system the layout does not take (unlike limbs)."""
    d = S.quadruped()
    sysm = brax(d)
    for N in (2000, 20000):
        st, a = inputs(sysm, d, N, 3)
        sysm.set_pair_launch(1, 1, 5)
        got = sysm.rollout(st, a)
        sysm.set_pair_launch(1, 1, 1)
        same(got, sysm.rollout(st, a))
    u = dict(d)
    u["stiffness"] = np.array(d["stiffness"]) * np.linspace(1.0, 0.9, len(d["stiffness"]))
    other = brax(u)
    from paper_2106_13281_gb300.binding import BraxError
    with pytest.raises(BraxError):
        other.set_pair_launch(1, 1, WIDE)
    other.rollout(*inputs(other, u, 100, 3))
    other.sync_status()


def ball_limbs(no_lower):
    """Two limbs whose lower bodies carry one point (a ball) or none."""
    sb = S.SceneBuilder()
    t = sb.body("torso", 10.0, S.UNIT_INERTIA, (0, 0, 0.75))
    sb.collider(t, S.CAPSULE, radius=0.25, length=0.5)
    ground = sb.plane()
    sb.pair(sb.collider_of(t), ground)
    for k, x in enumerate((-1.0, 1.0)):
        d = np.array([x, 0.0, 0.0])
        hip = np.array([0, 0, 0.75]) + 0.25 * d
        th = sb.capsule_body(f"thigh{k}", 1.0, 0.08, 0.4, hip + 0.2 * d, d, inertia=S.UNIT_INERTIA)
        sh = sb.body(f"foot{k}", 1.0, S.UNIT_INERTIA, hip + 0.5 * d)
        sb.collider(sh, S.CAPSULE, radius=0.1, length=0.2)
        jh = sb.joint(t, th, hip, axis=np.array([0.0, 1, 0]), ref=d, limits=((-40, 40),), **S.QUADRUPED_JOINT)
        sb.joint(th, sh, hip + 0.4 * d, axis=np.array([0.0, 1, 0]), ref=d, limits=((-40, 40),), **S.QUADRUPED_JOINT)
        sb.actuator(jh, 0, 100.0)
        sb.pair(sb.collider_of(th), ground)
        if not no_lower:
            sb.pair(sb.collider_of(sh), ground)
    return sb.build()


@pytest.mark.parametrize("no_lower", [False, True])
def test_limbs_with_other_point_counts(brax, no_lower):
    """Lower bodies of one point and of none: the wide kernel's counts at run time."""
    d = ball_limbs(no_lower)
    sysm = brax(d)
    st, a = inputs(sysm, d, 333, 40)
    sysm.set_pair_launch(1, 1, 1)
    ref = sysm.rollout(st, a, K=7, checkpoints=True, torso=True, contact_count=True)
    assert int(ref["contact_count"].sum()) > 0
    for v in (WIDE, SPLIT):
        sysm.set_pair_launch(1, 1, v)
        same(sysm.rollout(st, a, K=7, checkpoints=True, torso=True, contact_count=True), ref)
        sysm.sync_status()


def test_split_kernel_past_eight_warps_an_sm(brax):
    """The split kernel's launches on both sides of its two builds (7 and 9 warps
    an SM, 4 environments a warp)."""
    d = S.quadruped()
    sysm = brax(d)
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    for warps in (7, 9):
        st, a = inputs(sysm, d, 4 * warps * n_sm - 1, 6)
        sysm.set_pair_launch(1, 1, SPLIT)
        got = sysm.rollout(st, a, contact_count=True)
        sysm.set_pair_launch(1, 1, 1)
        same(got, sysm.rollout(st, a, contact_count=True))
        sysm.sync_status()
