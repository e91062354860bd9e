"""The matrix-product decode kernel at the edges of its arithmetic: integer sums next to the accumulator's 2^24, weights
whose reference has to move with nearly every tile, value scales spread over many binades; every container."""
import numpy as np
import pytest

from oracle import sa_oracle as ora
from paper_2609_09208_b200 import binding as sa
from paper_2609_09208_b200 import build as sa_build
from paper_2609_09208_b200 import synth

pytestmark = pytest.mark.gpu
CONTAINERS = [(0, False), (0, True), (1, False), (1, True), (2, True), (4, False), (8, False)]


def decode(case):
    import torch
    sa_build.build()
    dev = torch.device("cuda:0")
    up = lambda x: torch.from_numpy(np.ascontiguousarray(x).view(np.int16)).to(dev)
    cfg = sa.make_config(case.head_dim, case.n_q_heads, case.n_kv_heads, case.code_k, nibble=case.nibble)
    cache = sa.PagedCache(cfg, case.lens, dev)
    cache.fill(up(case.K), up(case.V), case.cu_lens)
    O = torch.full((case.batch, case.n_q_heads, case.head_dim), float("nan"), dtype=torch.float32, device=dev)
    dbg = torch.full((case.batch, case.n_q_heads, cache.max_pages * 64), -7, dtype=torch.int32, device=dev)
    sa.decode_attention(cfg, cache.handle, up(case.Q), O, cache.workspace, dbg)
    torch.cuda.synchronize()
    ref = ora.decode_attention(case.Q, case.K, case.V, case.cu_lens, case.code_k, 6 + (case.code_k if case.code_k != 8 else 0),
                               want_scores=True, n_threads=8)
    return O.cpu().numpy(), dbg.cpu().numpy(), ref


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("k,nibble", CONTAINERS)
def test_scores_exact_next_to_the_accumulator_limit(d, k, nibble):
    """Sums of terms of the largest magnitude with a few smallest ones in any position: every INT32 score as the oracle's."""
    rng = np.random.default_rng(100 + d + k)
    case = synth.make_case("limit", [333], 16, 2, d, k, nibble=nibble, seed=1)
    mags = np.array([1.0, 1.0, 1.0, 31 / 32, 2.0 ** -6, 17 / 16 * 2.0 ** -6, 0.0])
    K = rng.choice(mags, size=case.K.shape, p=[0.3, 0.3, 0.2, 0.1, 0.04, 0.03, 0.03])
    K[..., 0] = 1.0
    signs = rng.choice([-1.0, 1.0], size=case.K.shape)
    signs[::2] = 1.0                                          # half of the keys: all terms of one sign
    case.K[:] = (K * signs).astype(np.float16)
    Q = rng.choice([127.0, 126.0, 1.0], size=case.Q.shape, p=[0.9, 0.06, 0.04])
    Q[..., 1] = 127.0
    Q[:, 1::2] *= rng.choice([-1.0, 1.0], size=Q[:, 1::2].shape)
    case.Q[:] = Q.astype(np.float16)
    O, dbg, ref = decode(case)
    assert np.array_equal(dbg[0, :, :333].astype(np.int64), ref["A"][0])
    assert np.max(np.abs(O - ref["O"])) <= 1e-3


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("k,nibble", CONTAINERS)
@pytest.mark.parametrize("spread", [0, 6])
def test_outputs_with_a_moving_reference_and_spread_value_scales(d, k, nibble, spread):
    """Logits that grow along the sequence (the reference of the weights moves again and again) and value rows whose
    scales differ by up to 2^(2 * spread): outputs within 1e-5 of the oracle's in the 2-norm of every head."""
    rng = np.random.default_rng(200 + d + k)
    case = synth.make_case("moving", [700, 65], 8, 1, d, k, nibble=nibble, seed=3)
    q = case.Q[:, :1].astype(np.float32)
    case.Q[:] = (q * np.linspace(0.2, 1.0, 8)[None, :, None]).astype(np.float16)       # all heads look the same way
    for b in range(2):
        n = int(case.lens[b])
        ramp = np.linspace(-1.0, 3.0, n)[:, None, None]
        rows = slice(int(case.cu_lens[b]), int(case.cu_lens[b + 1]))
        case.K[rows] = (ramp * q[b][None] + 0.1 * case.K[rows]).astype(np.float16)
    case.V[:] = (case.V * np.exp2(rng.uniform(-spread, spread, (len(case.V), 1, 1)))).astype(np.float16)
    O, dbg, ref = decode(case)
    for b in range(2):
        assert np.array_equal(dbg[b, :, :case.lens[b]].astype(np.int64), ref["A"][b][:, :case.lens[b]])
        for h in range(8):
            err = np.linalg.norm(O[b, h] - ref["O"][b, h]) / np.linalg.norm(ref["O"][b, h])
            assert err <= 1e-5, (b, h, err)


@pytest.mark.parametrize("d,Hq,Hkv,lens", [(64, 32, 4, [0]), (64, 8, 1, [63]), (64, 32, 4, [1000]), (64, 1, 1, [2046]), (128, 8, 2, [1500]),
                                           (128, 16, 16, [200 + 7 * i for i in range(40)]), (64, 4, 4, [33] * 130)])
@pytest.mark.parametrize("k,nibble", [(0, True), (1, False), (4, False)])
def test_steps_without_a_merge_kernel(d, Hq, Hkv, lens, k, nibble):
    """Short single sequences (merged by a thread-block cluster) and batches with one split per sequence: several steps in
    a row without a synchronisation, the lengths counted up by the decode kernel itself; outputs as the oracle's on the
    extended cache, and as the same steps replayed from a CUDA graph."""
    import torch
    sa_build.build()
    dev = torch.device("cuda:0")
    up = lambda x: torch.from_numpy(np.ascontiguousarray(x).view(np.int16)).to(dev)
    lens, n_steps = np.asarray(lens), 3
    B = len(lens)
    full = synth.make_case("whole", lens + n_steps, Hq, Hkv, d, k, nibble=nibble, outliers=True, seed=300 + d + k)
    cfg = sa.make_config(d, Hq, Hkv, k, nibble=nibble)
    cache = sa.PagedCache(cfg, lens, dev, extra_tokens=n_steps)
    old = np.concatenate([np.arange(full.cu_lens[b], full.cu_lens[b] + lens[b]) for b in range(B)]).astype(np.int64)
    cache.fill(up(full.K[old]), up(full.V[old]), np.concatenate([[0], np.cumsum(lens)]))
    new = [np.array([full.cu_lens[b] + lens[b] + i for b in range(B)]) for i in range(n_steps)]
    Kn, Vn, Q = [up(full.K[n]) for n in new], [up(full.V[n]) for n in new], up(full.Q)
    O = [torch.full((B, Hq, d), float("nan"), dtype=torch.float32, device=dev) for _ in range(n_steps)]

    def steps():
        for i in range(n_steps):
            sa.decode_step(cfg, cache.handle, Q, Kn[i], Vn[i], O[i], cache.workspace)

    steps()
    torch.cuda.synchronize()
    assert cache.seq_lens.cpu().numpy().tolist() == (lens + n_steps).tolist()
    first = [o.clone() for o in O]
    for i in range(n_steps):
        rows = np.concatenate([np.arange(full.cu_lens[b], full.cu_lens[b] + lens[b] + i + 1) for b in range(B)])
        ref = ora.decode_attention(full.Q, full.K[rows], full.V[rows], np.concatenate([[0], np.cumsum(lens + i + 1)]), k, 6 + k,
                                   n_threads=8)["O"]
        assert np.max(np.abs(first[i].cpu().numpy() - ref)) <= 1e-3
    lens0 = torch.from_numpy(lens.astype(np.int32)).to(dev)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        cache.seq_lens.copy_(lens0)
        steps()
    for _ in range(2):
        for o in O:
            o.fill_(float("nan"))
        graph.replay()
        torch.cuda.synchronize()
        assert cache.seq_lens.cpu().numpy().tolist() == (lens + n_steps).tolist()
        assert all(torch.equal(a, b) for a, b in zip(O, first))


def one_launch_setup(lens, Hq, Hkv, d=64, k=4):
    import torch
    sa_build.build()
    dev = torch.device("cuda:0")
    up = lambda x: torch.from_numpy(np.ascontiguousarray(x).view(np.int16)).to(dev)
    lens = np.asarray(lens)
    B = len(lens)
    full = synth.make_case("arrive", lens + 1, Hq, Hkv, d, k, outliers=True, seed=330 + B)
    cfg = sa.make_config(d, Hq, Hkv, k)
    cache = sa.PagedCache(cfg, lens, dev, extra_tokens=1)
    old = np.concatenate([np.arange(full.cu_lens[b], full.cu_lens[b] + lens[b]) for b in range(B)]).astype(np.int64)
    cache.fill(up(full.K[old]), up(full.V[old]), np.concatenate([[0], np.cumsum(lens)]))
    new = np.array([full.cu_lens[b + 1] - 1 for b in range(B)])
    O = torch.full((B, Hq, d), float("nan"), dtype=torch.float32, device=dev)
    want = ora.decode_attention(full.Q, full.K, full.V, full.cu_lens, k, 6 + k, n_threads=8)["O"]
    return cfg, cache, up(full.Q), up(full.K[new]), up(full.V[new]), O, want


@pytest.mark.parametrize("lens,Hq,Hkv", [([1000], 32, 4), ([17], 1, 1), ([33] * 130, 4, 4)])
@pytest.mark.parametrize("contents", ["zeros", "ones", "random", "partials", "nearly the mark", "one below the mark"])
def test_step_of_one_launch_takes_a_workspace_with_any_contents(lens, Hq, Hkv, contents):
    """A step without a merge kernel counts its blocks in the workspace: the lengths grow by one whatever was there, and
    nothing behind the counting word is written (a step of two launches would leave its partials there)."""
    import torch
    cfg, cache, Q, K, V, O, want = one_launch_setup(lens, Hq, Hkv)
    ws, lens0 = cache.workspace, cache.seq_lens.clone()
    if contents == "zeros":
        ws.zero_()
    elif contents == "ones":
        ws.fill_(255)
    elif contents == "partials":
        sa.decode_attention(cfg, cache.handle, Q, O, ws, stages=1)
    else:
        ws.copy_(torch.randint(0, 256, ws.shape, generator=torch.Generator().manual_seed(5), dtype=torch.uint8))
        if contents == "nearly the mark":                    # its upper half, with other bits below
            ws[:8].view(torch.int64).copy_(torch.tensor([(0x7fa5c3d2 << 32) | (0x95 << 24) | 3]))
        if contents == "one below the mark":                 # the first block's addition makes the mark
            ws[:8].view(torch.int64).copy_(torch.tensor([(0x7fa5c3d296 << 24) - 1]))
    before = ws.clone()
    for i in range(3):
        cache.seq_lens.copy_(lens0)
        sa.decode_step(cfg, cache.handle, Q, K, V, O, ws)
        torch.cuda.synchronize()
        assert torch.equal(cache.seq_lens, lens0 + 1), i
        assert np.max(np.abs(O.cpu().numpy() - want)) <= 1e-3
    end = len(ws) - (16 if 2 <= len(lens) <= 128 else 0)
    assert torch.equal(ws[16:end], before[16:end])


def test_any_number_of_workspaces_serves_steps_of_one_launch():
    """A program with a workspace for every request, more than 4096 of them over its life: the last step is one launch as
    the first was, from a side stream and recorded in a graph before any other call too."""
    import torch
    cfg, cache, Q, K, V, O, want = one_launch_setup([300], 8, 1)
    lens0 = cache.seq_lens.clone()
    size = (len(cache.workspace) + 255) // 256 * 256
    pool = torch.full((4200, size), 255, dtype=torch.uint8, device="cuda")
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        cache.seq_lens.copy_(lens0)
        sa.decode_step(cfg, cache.handle, Q, K, V, O, pool[0])
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(cache.seq_lens, lens0 + 1)
    with torch.cuda.stream(torch.cuda.Stream()):
        for ws in pool[1:]:
            cache.seq_lens.copy_(lens0)
            sa.decode_step(cfg, cache.handle, Q, K, V, O, ws)
    torch.cuda.synchronize()
    assert torch.equal(cache.seq_lens, lens0 + 1)
    assert np.max(np.abs(O.cpu().numpy() - want)) <= 1e-3
    assert bool((pool[:, 16:] == 255).all())


@pytest.mark.parametrize("lens,lost", [([2000], (0, 1, 40)), ([2000], (0, 3, 62)), ([70], (0, 0, 2)), ([20], (0, 2, 0)), ([33, 64, 0, 5], (1, 2, 1))])
def test_lost_copy_is_marked_where_no_merge_kernel_runs(lens, lost):
    """The bounded wait of a copy made to run out (test hook, 2^10 polls) where the splits of a sequence are merged in their
    thread-block cluster or the sequence has one split: exactly the rows of that (sequence, KV head) are NaN, the others
    ordinary, and the call was one launch (no partials behind)."""
    import torch
    sa_build.build()
    dev = torch.device("cuda:0")
    up = lambda x: torch.from_numpy(np.ascontiguousarray(x).view(np.int16)).to(dev)
    b, kvh, tile = lost
    case = synth.make_case("lost", lens, 32, 4, 64, 4, outliers=True, seed=5200)
    cfg = sa.make_config(64, 32, 4, sa.SA_POTM4)
    cache = sa.PagedCache(cfg, case.lens, dev)
    cache.fill(up(case.K), up(case.V), case.cu_lens)
    O = torch.zeros((case.batch, 32, 64), dtype=torch.float32, device=dev)
    cache.workspace.fill_(255)
    sa.debug_decode_lost_copy(cfg, cache.handle, up(case.Q), O, cache.workspace, b, kvh, tile)
    torch.cuda.synchronize()
    got = O.cpu().numpy()
    ref = ora.decode_attention(case.Q, case.K, case.V, case.cu_lens, 4, 10, n_threads=8)["O"]
    hit = np.zeros((case.batch, 32), dtype=bool)
    hit[b, kvh * 8:(kvh + 1) * 8] = True
    assert np.isnan(got[hit]).all()
    assert np.max(np.abs(got[~hit] - ref[~hit])) <= 1e-3
    end = len(cache.workspace) - (16 * ((8 * case.batch + 15) // 16) if case.batch > 1 else 0)
    assert bool((cache.workspace[:end] == 255).all())


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("k,nibble", CONTAINERS + [(16, False)])
@pytest.mark.parametrize("size,sign", [(2000, 1), (3000, 1), (4000, 1), (6000, -1)])
def test_logits_beyond_the_integers_of_a_float(d, k, nibble, size, sign):
    """Keys and queries whose logits reach 2^25.4 .. 2^27.9 in the log2 domain, where a float near the reference is off by
    more than the weights have to spare, growing along the sequence so that the reference moves often, or all of them far below zero:
    every row is the value row of its best key (the next best is 1024 or more below), with scales 2^-8 .. 2^8."""
    import torch
    sa_build.build()
    dev = torch.device("cuda:0")
    up = lambda x: torch.from_numpy(np.ascontiguousarray(x).view(np.int16)).to(dev)
    rng = np.random.default_rng(400 + d + k + size)
    lens = [900] if size == 3000 else [900, 65]  # one sequence: merged in a cluster
    case = synth.make_case("large", lens, 8, 1, d, 0 if k == 16 else k, nibble=nibble, seed=5)
    pattern = rng.choice([-1.0, 1.0], size=d)
    case.Q[:] = (size * np.linspace(0.5, 1.0, 8)[None, :, None] * pattern).astype(np.float16)
    for b in range(len(lens)):
        rows = slice(int(case.cu_lens[b]), int(case.cu_lens[b + 1]))
        ramp = np.linspace(0.3, 1.0, int(case.lens[b])) if sign > 0 else np.linspace(1.0, 0.3, int(case.lens[b]))
        case.K[rows] = (sign * size * ramp[:, None, None] * pattern).astype(np.float16)
        case.K[rows.stop - 2] = case.K[rows.stop - 1] / 2     # (the ends of the ramp are apart in binary16 too)
    case.V[:] = (case.V * np.exp2(rng.uniform(-8, 8, (len(case.V), 1, 1)))).astype(np.float16)
    cfg = sa.make_config(d, 8, 1, k, nibble=nibble)
    cache = sa.PagedCache(cfg, case.lens, dev)
    cache.fill(up(case.K), up(case.V), case.cu_lens)
    O = torch.zeros((len(lens), 8, d), dtype=torch.float32, device=dev)
    (sa.decode_attention_fp16 if k == 16 else sa.decode_attention)(cfg, cache.handle, up(case.Q), O, cache.workspace)
    torch.cuda.synchronize()
    O = O.cpu().numpy()
    assert np.isfinite(O).all()
    for b in range(len(lens)):
        rows = slice(int(case.cu_lens[b]), int(case.cu_lens[b + 1]))
        score = case.K[rows, 0].astype(np.float64) @ pattern
        z = np.sort(score)[::-1] * size * 0.5 / np.sqrt(d) * 1.4427
        assert z[0] - z[1] >= 1024
        best = case.V[rows, 0][np.argmax(score)]
        vhat, g = ora.quantise_value(best[None])
        want = best.astype(np.float64) if k == 16 else vhat[0] * 2.0 ** -float(g[0])
        err = np.linalg.norm(O[b] - want, axis=1) / np.linalg.norm(want)
        assert err.max() <= 1e-5, (b, err)
