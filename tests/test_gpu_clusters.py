"""Batches of short sequences: one thread-block cluster per (sequence, KV head), and their steps from host buffers, whose inputs
one block of each cluster fetches."""
import numpy as np
import pytest

from oracle import sa_oracle as ora
from paper_2609_09208_b200 import binding as sa
from paper_2609_09208_b200 import build as sa_build
from paper_2609_09208_b200 import synth

pytestmark = pytest.mark.gpu
# the fewest units and the most; one tile a block, clusters of 4, several rounds; every shape of block
SHAPES = [(64, 32, 4, sa.SA_POTM1, True, [0, 33]), (64, 32, 4, sa.SA_POT4, True, [2111, 1, 64, 700]), (64, 32, 4, sa.SA_POTM4, False, [200, 0, 31, 32, 33, 500, 64, 65]),
          (64, 32, 4, sa.SA_POTM2, False, [6000, 5, 2000, 64, 0, 1, 900, 95]), (64, 1, 1, sa.SA_POT4, False, [(67 * i) % 1000 for i in range(32)]),
          (128, 32, 8, sa.SA_POTM4, False, [3000, 64]), (128, 16, 16, sa.SA_POTM2, True, [700, 0]), (64, 32, 4, sa.SA_KV_FP16, False, [3000, 31, 0, 64])]


@pytest.mark.parametrize("d,Hq,Hkv,code,dense,lens", SHAPES)
def test_steps_of_short_batches_from_device_and_host_buffers(d, Hq, Hkv, code, dense, lens):
    """Three steps in one launch each (the partials' part of the workspace stays as it was), outputs as the oracle's; from pinned
    host buffers the same bits and the same cache."""
    import torch
    sa_build.build()
    up = lambda x: torch.from_numpy(np.ascontiguousarray(x).view(np.int16)).cuda()
    lens, n, B = np.asarray(lens), 3, len(lens)
    k = 0 if code == sa.SA_KV_FP16 else code
    full = synth.make_case("cluster", lens + n, Hq, Hkv, d, k, nibble=dense, outliers=True, seed=8400 + d + B)
    cfg = sa.make_config(d, Hq, Hkv, code, nibble=dense)
    old = np.concatenate([np.arange(full.cu_lens[b], full.cu_lens[b] + lens[b]) for b in range(B)]).astype(np.int64)
    caches = []
    for _ in range(2):
        c = sa.PagedCache(cfg, lens, "cuda", extra_tokens=n)
        c.fill(up(full.K[old]), up(full.V[old]), np.concatenate([[0], np.cumsum(lens)]))
        c.workspace.fill_(255)
        caches.append(c)
    staging = torch.empty(sa.staging_bytes(cfg, B), dtype=torch.uint8, device="cuda")
    Q = up(full.Q)
    for i in range(n):
        new = np.array([full.cu_lens[b] + lens[b] + i for b in range(B)])
        K, V = up(full.K[new]), up(full.V[new])
        O = torch.full((B, Hq, d), float("nan"), device="cuda")
        Oh = torch.full((B, Hq, d), float("nan")).pin_memory()
        sa.decode_step(cfg, caches[0].handle, Q, K, V, O, caches[0].workspace)
        sa.decode_step_host(cfg, caches[1].handle, *[x.cpu().pin_memory() for x in (Q, K, V)], Oh, staging, caches[1].workspace)
        torch.cuda.synchronize()
        rows = np.concatenate([np.arange(full.cu_lens[b], full.cu_lens[b] + lens[b] + i + 1) for b in range(B)])
        cu = np.concatenate([[0], np.cumsum(lens + i + 1)])
        if code == sa.SA_KV_FP16:
            want = np.stack([ora.sdpa_fp16(full.Q[b], full.K[rows[cu[b]:cu[b + 1]]], full.V[rows[cu[b]:cu[b + 1]]]) for b in range(B)])
        else:
            want = ora.decode_attention(full.Q, full.K[rows], full.V[rows], cu, k, 6 + k, n_threads=8)["O"]
        assert np.max(np.abs(O.cpu().numpy() - want)) <= 1e-3
        assert torch.equal(O.cpu(), Oh)
        assert torch.equal(caches[0].pages, caches[1].pages) and torch.equal(caches[0].seq_lens, caches[1].seq_lens)
        assert caches[0].seq_lens.cpu().numpy().tolist() == (lens + i + 1).tolist()
    end = len(caches[0].workspace) - 16 * ((8 * B + 15) // 16)
    assert bool((caches[0].workspace[16:end] == 255).all())
