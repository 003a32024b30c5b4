"""Chunked rollouts of one system on more streams at once than it has scheduler
regions, beside a replaying CUDA graph: every result is the static schedule's."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2106_13281_gb300 import scenes as S

pytestmark = pytest.mark.gpu


def test_concurrent_chunked_rollouts_and_a_graph():
    from paper_2106_13281_gb300.system import BraxSystem
    d = S.quadruped()
    sysm = BraxSystem(d)
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    N, T, lanes = 2 * n_sm * 64 + 640, 40, 7  # ten blocks past one wave of the wide limb kernel
    rp, rr, ang = S.initial_conditions(d, N, 61, height_jitter=0.05)
    f32 = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()
    st = sysm.default_qp(N, f32(rp), f32(rr), f32(ang))
    acts = [f32(S.actions(d, N, T, 62 + i)) for i in range(lanes + 1)]
    sysm.set_schedule(0)
    ref = [sysm.rollout(st, a)["state_T"] for a in acts]
    short = sysm.rollout(st, acts[0][:20])["state_T"]
    sysm.set_schedule(1)
    assert torch.equal(sysm.rollout(st, acts[0])["state_T"], ref[0])
    assert sysm.last_rollout()["n_chunks"] > 1
    torch.cuda.synchronize()

    side, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side):
        got_short = sysm.rollout(st, acts[lanes][:20])
        assert sysm.last_rollout()["n_chunks"] == 0  # too short to be cut in a captured launch
        got_graph = sysm.rollout(st, acts[lanes])
        assert sysm.last_rollout()["n_chunks"] > 1
    streams = [torch.cuda.Stream() for _ in range(lanes)]
    outs = [torch.empty_like(st) for _ in range(3 * lanes)]
    shorts = [torch.empty_like(st) for _ in range(lanes)]
    torch.cuda.synchronize()
    for r in range(3):
        with torch.cuda.stream(side):
            graph.replay()
        for i, s in enumerate(streams):
            with torch.cuda.stream(s):
                sysm.rollout(st, acts[i], state_T=outs[3 * i + r])
    for i, s in enumerate(streams):
        with torch.cuda.stream(s):
            sysm.rollout(st, acts[0][:20], state_T=shorts[i])
            assert sysm.last_rollout()["n_chunks"] > 1
    torch.cuda.synchronize()
    sysm.sync_status()
    for i in range(lanes):
        for r in range(3):
            assert torch.equal(outs[3 * i + r], ref[i]), (i, r)
        assert torch.equal(shorts[i], short)
    assert torch.equal(got_graph["state_T"], ref[lanes])
    assert bool(torch.isfinite(got_short["state_T"]).all())
