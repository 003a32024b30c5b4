"""The default block size of a heterogeneous batch of more blocks than are
resident at once, where warp slots alone would ask for more groups a block than
its shared memory holds: forward and reverse run, and each system's slice equals
its solo launch (the tolerances of test_gpu_batch.py)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2106_13281_gb300 import scenes as S

pytestmark = pytest.mark.gpu


def chain(n, pairs=0):
    """A hinge chain of n bodies, each with three capsules; the first `pairs`
    pairs of capsules of bodies at least two apart are tested (at most 24 a
    body, as the library takes them)."""
    sb = S.SceneBuilder()
    cols, prev = [], None
    for i in range(n):
        b = sb.body(f"b{i}", 1.0, S.UNIT_INERTIA, (0.3 * i, 0, 1.0))
        cols.append([sb.collider(b, S.CAPSULE, pos=(0, 0.1 * k - 0.1, 0), radius=0.04, length=0.2) for k in range(3)])
        if prev is not None:
            j = sb.joint(prev, b, (0.3 * i - 0.15, 0, 1.0), axis=(0, 1, 0), ref=(1, 0, 0), limits=((-60, 60),),
                         **S.QUADRUPED_JOINT)
            sb.actuator(j, 0, 5.0)
        prev = b
    used = [0] * n
    for k in range(9):
        for a in range(n):
            for b in range(a + 2, n):
                if len(sb.pairs) < pairs and max(used[a], used[b]) < 24:
                    sb.pair(cols[a][k // 3], cols[b][k % 3])
                    used[a] += 1
                    used[b] += 1
    assert len(sb.pairs) == pairs
    return sb.build()


SETS = {
    # 32 warps by warp slots; the reverse of two 16-body groups takes 278,784 bytes
    "20 + 16 bodies": lambda: [(chain(20), 64), (chain(16), 8192)],
    # 27 warps by warp slots; the reverse of three quadruped groups takes 235,392 bytes
    "20 bodies + quadruped": lambda: [(chain(20), 32), (S.quadruped(), 16384)],
    # 18 warps by warp slots; the forward of two 9-body groups of 100 pairs takes 255,232 bytes
    "17 + 9 bodies, pairs": lambda: [(chain(17, 20), 32), (chain(9, 100), 8192)],
}


@pytest.mark.parametrize("name", list(SETS))
def test_large_blocks_fit_and_match_solo(name):
    from paper_2106_13281_gb300.system import BraxBatch, BraxSystem
    descs, n = zip(*SETS[name]())
    systems = [BraxSystem(d) for d in descs]
    for s in systems:
        if s.paired:
            s.set_pair_launch(0, 1, 0)
    T, K = 2, 2
    f32 = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()
    parts = []
    for s, m in zip(systems, n):
        rp, rr, ang = S.initial_conditions(s.desc, m, 51, height_jitter=0.05)
        st = s.default_qp(m, f32(rp), f32(rr), f32(ang))
        parts.append((st, f32(S.actions(s.desc, m, T, 52)), torch.ones_like(st)))
    st, a, g = (torch.cat([p[i].flatten() for p in parts]) for i in range(3))
    batch = BraxBatch(systems, n)
    out = batch.rollout(st, a, T, K=K, checkpoints=True)
    ga, gs = batch.rollout_backward(st, a, out["checkpoints"], g, T, K=K)
    for i, (s, m) in enumerate(zip(systems, n)):
        so, ao, _, _ = batch.offsets(T, K, i)
        solo = s.rollout(parts[i][0], parts[i][1], K=K, checkpoints=True)
        ra, rs = s.rollout_backward(parts[i][0], parts[i][1], solo["checkpoints"], parts[i][2], K=K)
        close = lambda x, y, scale: torch.allclose(x.view(y.shape), y, rtol=1e-4, atol=1e-5 * scale)
        assert torch.allclose(out["state_T"][so:so + rs.numel()].view(rs.shape), solo["state_T"], rtol=1e-6, atol=1e-6)
        assert close(gs[so:so + rs.numel()], rs, rs.abs().max().item() + 1.0)
        assert close(ga[ao:ao + ra.numel()], ra, ra.abs().max().item() + 1.0)
        s.sync_status()


def test_a_refused_launch_leaves_no_error_behind():
    """The reverse pass of 28 bodies needs more shared memory than a block has
    and is refused with an error code; the next call runs."""
    from paper_2106_13281_gb300.binding import BraxError
    from paper_2106_13281_gb300.system import BraxSystem
    s = BraxSystem(chain(28))
    st = s.default_qp(32)
    a = torch.zeros((1, 32, s.A), device="cuda")
    ck = s.rollout(st, a, K=1, checkpoints=True)["checkpoints"]
    with pytest.raises(BraxError):
        s.rollout_backward(st, a, ck, torch.ones_like(st), K=1)
    assert torch.equal(s.default_qp(32), st)
    s.sync_status()
