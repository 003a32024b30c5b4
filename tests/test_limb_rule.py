"""Which kernel the default launch of a limb-layout system takes, by its number
of limbs, environments (as warps of the split kernel an SM), steps and the
environment layer; and, on the GPU, that the default launch gives the paired
body-layout kernel's bits at each of these sizes."""
import ctypes as C

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2106_13281_gb300 import scenes as S

SPLIT, WIDE, BODY = 7, 6, 0
# limbs, warps an SM, steps, environment layer, kernel
RULE = [
    (1, 3, 2, False, SPLIT), (1, 6, 2, False, BODY), (1, 10, 16, False, WIDE), (1, 10, 15, False, BODY),
    (1, 10, 20, True, BODY), (1, 14, 4, False, WIDE), (1, 14, 3, False, BODY), (1, 14, 4, True, BODY),
    (1, 20, 2, False, BODY), (1, 30, 1, False, WIDE), (1, 33, 1, False, BODY), (1, 33, 2, False, WIDE),
    (1, 33, 2, True, WIDE), (2, 10, 2, True, SPLIT), (2, 14, 2, True, WIDE), (2, 18, 2, False, SPLIT),
    (2, 23, 2, True, BODY), (2, 30, 1, True, WIDE), (2, 33, 1, True, BODY), (2, 40, 1, False, BODY),
    (2, 41, 1, False, WIDE), (4, 7, 1, True, SPLIT), (4, 12, 1, False, WIDE), (4, 18, 1, True, SPLIT),
    (4, 24, 1, False, WIDE), (4, 33, 1, True, WIDE), (8, 33, 1, False, WIDE),
]


def n_envs(limbs, warps, n_sm):
    return warps * n_sm * (16 // limbs)


@pytest.mark.parametrize("limbs,warps,T,env,kernel", RULE)
def test_rule(limbs, warps, T, env, kernel):
    from paper_2106_13281_gb300 import binding, build
    build.build()
    f = binding.load_library().brax_internal_limb_rule
    f.argtypes = [C.c_int32, C.c_int64, C.c_int32, C.c_int32, C.c_int32]
    for n_sm in (152, 148):
        N = n_envs(limbs, warps, n_sm)
        assert f(limbs, N, T, int(env), n_sm) == kernel
        assert f(limbs, N - 1, T, int(env), n_sm) == kernel


@pytest.mark.gpu
@pytest.mark.parametrize("limbs,warps,T,env,kernel", [r for r in RULE if r[0] < 8])
def test_default_launch_gives_the_paired_bits(limbs, warps, T, env, kernel):
    from paper_2106_13281_gb300.system import BraxSystem
    from test_gpu_limb import crawler
    d = {1: S.pendulum, 2: lambda: crawler(2), 4: S.quadruped}[limbs]()
    N = n_envs(limbs, warps, torch.cuda.get_device_properties(0).multi_processor_count) - 1
    default, paired = BraxSystem(d), BraxSystem(d)
    paired.set_pair_launch(1, 1, 1)
    rp, rr, ang = S.initial_conditions(d, N, 71, height_jitter=0.05)
    if limbs > 1:
        rp[:, 2] -= 0.36  # on the ground
    f32 = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()
    st, a = default.default_qp(N, f32(rp), f32(rr), f32(ang)), f32(S.actions(d, N, T, 72))
    if env:
        got, ref = (s.env_rollout(st, a, min_z=0.3, max_z=0.8) for s in (default, paired))
    else:
        got, ref = (s.rollout(st, a, K=2, checkpoints=True, torso=True, contact_count=True) for s in (default, paired))
    for k in ref:
        assert torch.equal(got[k], ref[k]), k
    default.sync_status()
