"""The reverse pass stays inside the workspace that the size calls ask for: the
bytes behind it are untouched, also when the checkpoint interval is longer than
the rollout."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2106_13281_gb300 import scenes as S

pytestmark = pytest.mark.gpu

GUARD = 1 << 20
NAMES = ("pendulum", "quadruped", "biped")


@pytest.fixture(scope="module")
def systems():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2106_13281_gb300.system import BraxSystem
    return [BraxSystem(S.SCENES[n]()) for n in NAMES]


def inputs(s, N, T):
    rp, rr, ang = S.initial_conditions(s.desc, N, 7, height_jitter=0.05)
    f32 = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()
    return s.default_qp(N, f32(rp), f32(rr), f32(ang)), f32(S.actions(s.desc, N, T, 8))


def guarded(need):
    """A workspace of exactly `need` bytes, and the guarded array it lies in."""
    big = torch.full((need + GUARD,), 0xA5, device="cuda", dtype=torch.uint8)
    return big[:need], big


@pytest.mark.parametrize("T,K", [(1, 10), (2, 10), (3, 2)])
def test_reverse_pass_stays_inside_its_workspace(systems, T, K):
    s, N = systems[1], 70
    st, a = inputs(s, N, T)
    ck = s.rollout(st, a, K=K, checkpoints=True)["checkpoints"]
    need = s.workspace_size(N, T, K)
    ws, big = guarded(need)
    got = s.rollout_backward(st, a, ck, torch.ones_like(st), K=K, workspace=ws)
    s.sync_status()
    assert bool((big[need:] == 0xA5).all())
    ref = s.rollout_backward(st, a, s.rollout(st, a, K=1, checkpoints=True)["checkpoints"], torch.ones_like(st), K=1)
    assert torch.equal(got[0], ref[0]) and torch.equal(got[1], ref[1])


def batch_of(systems, T, K):
    from paper_2106_13281_gb300.system import BraxBatch
    n = [40, 70, 33][:len(systems)]
    b = BraxBatch(systems, n)
    parts = [inputs(s, m, T) for s, m in zip(systems, n)]
    st, a = torch.cat([p[0].flatten() for p in parts]), torch.cat([p[1].flatten() for p in parts])
    return b, st, a, b.rollout(st, a, T, K=K, checkpoints=True)["checkpoints"]


@pytest.mark.parametrize("T,K", [(1, 10), (2, 5), (5, 2)])
def test_batch_reverse_pass_stays_inside_its_workspace(systems, T, K):
    b, st, a, ck = batch_of(systems, T, K)
    need = b.workspace_size(T, K)
    ws, big = guarded(need)
    b.rollout_backward(st, a, ck, torch.ones_like(st), T, K=K, workspace=ws)
    for s in systems:
        s.sync_status()
    assert bool((big[need:] == 0xA5).all())


@pytest.mark.parametrize("names", [("pendulum", "quadruped"), ("quadruped", "biped")])
@pytest.mark.parametrize("T,K", [(5, 2), (4, 4)])
def test_batch_gradients_do_not_depend_on_the_workspace(systems, names, T, K):
    """The size asked for (all substep states of a segment) and a smaller one
    (step states, substeps recomputed): the same bits, for hinge-only systems
    and for general ones; less still is refused."""
    from paper_2106_13281_gb300.binding import _ptr, _stream
    sub = [s for s, n in zip(systems, NAMES) if n in names]
    b, st, a, ck = batch_of(sub, T, K)
    need = b.workspace_size(T, K)
    g = torch.ones_like(st)
    outs = []
    for nbytes in (need, need - 1):
        ws, big = guarded(nbytes)
        ga, gs = torch.empty_like(a), torch.empty_like(st)
        args = (b._h, T, K, _ptr(st), _ptr(a), _ptr(ck), _ptr(g), None, _ptr(ga), _ptr(gs), _ptr(ws))
        assert b._L.brax_batch_rollout_backward(*args, nbytes, _stream()) == 0
        torch.cuda.synchronize()
        assert bool((big[nbytes:] == 0xA5).all())
        outs.append((ga, gs))
        assert b._L.brax_batch_rollout_backward(*args, 4096, _stream()) == 7
    assert torch.equal(outs[0][0], outs[1][0]) and torch.equal(outs[0][1], outs[1][1])


def test_a_smaller_batch_workspace_is_used(systems):
    """BraxBatch.rollout_backward runs in a smaller workspace than it asks for
    instead of allocating the full one, and replaces one too small to run in."""
    T, K = 4, 4
    b, st, a, ck = batch_of(systems, T, K)
    g, need = torch.ones_like(st), b.workspace_size(T, K)
    ref = b.rollout_backward(st, a, ck, g, T, K=K)
    for nbytes, allocates in ((need - 256, False), (256, True)):
        ws = torch.empty(nbytes, device="cuda", dtype=torch.uint8)
        torch.cuda.synchronize()
        torch.cuda.reset_peak_memory_stats()
        before = torch.cuda.memory_allocated()
        got = b.rollout_backward(st, a, ck, g, T, K=K, workspace=ws)
        assert (torch.cuda.max_memory_allocated() - before >= need) == allocates
        assert torch.equal(got[0], ref[0]) and torch.equal(got[1], ref[1])
