"""Forms of a decode step and of a call that the other tests do not reach: host buffers in front of every kernel, more sequences
than a warp has lanes, and one workspace for calls of different forms."""
import numpy as np
import pytest

from paper_2609_09208_b200 import binding as sa
from paper_2609_09208_b200 import build as sa_build
from paper_2609_09208_b200 import synth
from test_gpu_stream import MIX, attend, marks, up, wide_cache

pytestmark = pytest.mark.gpu
# head_dim, query heads, KV heads, code, lengths, tokens the page table has room for (0: what the lengths need), whether the call goes to
# the kernel of one block per SM: behind the staging kernel; inputs fetched by a block that is no cluster (one page, or one split of more than
# 128 sequences); clusters
FORMS = [(64, 32, 4, sa.SA_POTM4, MIX, 16384, True), (128, 32, 8, sa.SA_POTM4, MIX, 8192, True),
         (64, 8, 1, sa.SA_POTM4, [(37 * i) % 400 for i in range(128)], 8192, True), (64, 32, 4, sa.SA_KV_FP16, MIX * 3, 16384, True),
         (64, 8, 1, sa.SA_POTM1, [10], 0, False), (128, 4, 4, sa.SA_KV_FP16, [0], 0, False), (64, 4, 4, sa.SA_POTM4, [(7 * i) % 62 for i in range(130)], 0, False),
         (64, 32, 4, sa.SA_POT4, [100, 64, 0, 31], 0, False)]


@pytest.mark.parametrize("d,Hq,Hkv,code,lens,room,stream", FORMS)
def test_steps_from_device_and_host_buffers_equal_append_and_decode(d, Hq, Hkv, code, lens, room, stream):
    """Three steps, as calls and replayed from a graph: bytes, lengths and outputs."""
    import torch
    sa_build.build()
    lens, n, B = np.asarray(lens), 3, len(lens)
    full = synth.make_case("forms", lens + n, Hq, Hkv, d, 0 if code == sa.SA_KV_FP16 else code, outliers=True, seed=8800 + d + B)
    cfg = sa.make_config(d, Hq, Hkv, code)
    old = np.concatenate([np.arange(full.cu_lens[b], full.cu_lens[b] + lens[b]) for b in range(B)]).astype(np.int64)
    room = room or (int(lens.max()) + n + 63) // 64 * 64
    caches = [wide_cache(cfg, lens, room, extra=n) for _ in range(3)]
    for c in caches:
        c.fill(up(full.K[old]), up(full.V[old]), np.concatenate([[0], np.cumsum(lens)]))
    ref, step, host = caches
    lens0 = ref.seq_lens.clone()
    new = [np.array([full.cu_lens[b] + lens[b] + i for b in range(B)]) for i in range(n)]
    Q, K, V = up(full.Q), [up(full.K[x]) for x in new], [up(full.V[x]) for x in new]
    pin = lambda x: x.cpu().pin_memory()
    Qh, Kh, Vh = pin(Q), [pin(x) for x in K], [pin(x) for x in V]
    staging = torch.full((sa.staging_bytes(cfg, B),), 255, dtype=torch.uint8, device="cuda")
    O = [[torch.full((B, Hq, d), float("nan"), device="cuda") for _ in range(n)] for _ in range(2)]
    Oh = [pin(o) for o in O[0]]
    for i in range(n):
        sa.append_kv(cfg, ref.handle, K[i], V[i], True)
        attend(cfg, ref, Q, O[0][i])

    def steps():
        for i in range(n):
            sa.decode_step(cfg, step.handle, Q, K[i], V[i], O[1][i], step.workspace)
            sa.decode_step_host(cfg, host.handle, Qh, Kh[i], Vh[i], Oh[i], staging, host.workspace)

    steps()
    torch.cuda.synchronize()
    assert (marks(step.workspace) > 1) == stream
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        step.seq_lens.copy_(lens0)
        host.seq_lens.copy_(lens0)
        steps()
    for replay in range(3):
        for c in (step, host):
            assert torch.equal(c.pages, ref.pages) and torch.equal(c.seq_lens, lens0 + n) and torch.equal(c.seq_lens, ref.seq_lens)
        for i in range(n):
            assert torch.equal(O[1][i], O[0][i]) and torch.equal(Oh[i], O[0][i].cpu())
            O[1][i].fill_(float("nan"))
            Oh[i].fill_(float("nan"))
        if replay < 2:
            graph.replay()
            torch.cuda.synchronize()


def test_one_workspace_for_calls_of_different_forms_in_turn():
    """Units across blocks, a cluster per unit, one split and partials with a merge kernel, each after every other, nothing waited for."""
    import torch
    sa_build.build()
    forms = [(64, 32, 4, sa.SA_POTM4, MIX, 16384), (64, 32, 4, sa.SA_POT4, [700, 64, 0, 31], 0), (64, 4, 4, sa.SA_POTM4, [33] * 130, 0),
             (128, 32, 8, sa.SA_POTM1, [20000], 0), (128, 32, 8, sa.SA_POTM4, MIX, 8192)]
    calls = []
    for d, Hq, Hkv, code, lens, room in forms:
        lens = np.asarray(lens)
        case = synth.make_case("turn", lens, Hq, Hkv, d, code, seed=8900 + d + len(lens))
        cfg = sa.make_config(d, Hq, Hkv, code)
        c = wide_cache(cfg, lens, room or (int(lens.max()) + 64) // 64 * 64, extra=1)
        c.fill(up(case.K), up(case.V), case.cu_lens)
        new = [up(x[np.minimum(np.arange(len(lens)), len(x) - 1)]) for x in (case.K, case.V)]
        calls.append((cfg, c, up(case.Q), new, c.seq_lens.clone()))

    def run(call, workspace):
        cfg, c, Q, (K, V), lens0 = call
        O = torch.full(Q.shape, float("nan"), device="cuda")
        c.seq_lens.copy_(lens0)
        sa.decode_step(cfg, c.handle, Q, K, V, O, workspace)
        return O, c.seq_lens.clone()

    want = [run(call, call[1].workspace) for call in calls]
    one = torch.full((max(len(call[1].workspace) for call in calls),), 255, dtype=torch.uint8, device="cuda")
    order = [b for a in range(5) for i in range(5) for b in (a, i)]
    got = [(i, run(calls[i], one)) for i in order]
    torch.cuda.synchronize()
    for i, (O, lens) in got:
        assert torch.equal(O, want[i][0]) and torch.equal(lens, want[i][1]) and torch.equal(lens, calls[i][4] + 1), i
