"""The decode kernel of one block per SM: stretches of tiles cut across sequences and query groups, at the edges of units.

It serves calls whose cache has room for much work; the room is in the page table, so short sequences go through it here,
whose units lie many to a block, in one block alone, or across several."""
import numpy as np
import pytest

from oracle import sa_oracle as ora
from paper_2609_09208_b200 import binding as sa
from paper_2609_09208_b200 import build as sa_build
from paper_2609_09208_b200 import synth

pytestmark = pytest.mark.gpu
MARK = 0x7fa5c3d296                               # the upper 40 bits of a counting word at rest
EDGES = [0, 1, 31, 32, 33, 63, 64, 65]
MIX = EDGES + [700, 0, 95, 5000, 2, 333, 1111, 96]
# head_dim, query heads, KV heads, code, dense container, rotation, lengths, tokens the page table has room for
SHAPES = [
    (64, 32, 4, sa.SA_POTM4, False, False, MIX, 16384), (64, 32, 4, sa.SA_POT4, True, True, MIX[::-1], 16384),
    (64, 32, 4, sa.SA_POTM1, True, False, [777] * 37, 8192), (64, 32, 4, sa.SA_INT8, False, False, MIX * 2, 8192),
    (64, 16, 1, sa.SA_POTM2, False, False, MIX * 2, 16384),                # two blocks' worth of query heads per KV head
    (64, 8, 1, sa.SA_POTM4, False, False, [(37 * i) % 400 for i in range(128)], 8192),
    (64, 5, 5, sa.SA_POTM2, True, False, MIX * 2, 16384), (128, 32, 8, sa.SA_POTM4, False, False, MIX, 8192),
    (128, 64, 8, sa.SA_POTM1, False, False, MIX, 8192),                   # rows that have no place of their own in shared memory
    (128, 16, 16, sa.SA_POTM2, True, True, MIX[:8] * 2, 8192), (64, 32, 4, sa.SA_KV_FP16, False, False, MIX * 2, 16384),
    (128, 32, 8, sa.SA_KV_FP16, False, False, MIX * 2, 16384)]


def up(x):
    import torch
    return torch.from_numpy(np.ascontiguousarray(x).view(np.int16)).cuda()


def wide_cache(cfg, lens, room, extra=0, seed=5):
    """A cache of these lengths whose page table has `room` tokens a sequence, and a workspace for that."""
    import torch
    n_pages = int(np.maximum((np.asarray(lens) + extra + 63) // 64, 1).sum())
    c = sa.PagedCache(cfg, lens, "cuda", extra_tokens=extra, permutation=synth.page_permutation(n_pages, seed))
    table = torch.full((len(lens), room // 64), -1, dtype=torch.int32, device="cuda")
    table[:, :c.max_pages] = c.page_table
    c.page_table, c.max_pages = table, room // 64
    c.handle = sa.make_cache(c.pages, table, c.seq_lens, c.n_pages)
    c.workspace = torch.full((sa.workspace_bytes(cfg, len(lens), room // 64),), 255, dtype=torch.uint8, device="cuda")
    return c


def marks(ws):
    words = ws[:len(ws) // 8 * 8].cpu().numpy().view(np.uint64)
    return int(((words >> 24) == MARK).sum())


def attend(cfg, c, Q, O, dbg=None, stages=3):
    if cfg.code == sa.SA_KV_FP16:
        sa.decode_attention_fp16(cfg, c.handle, Q, O, c.workspace, stages)
    else:
        sa.decode_attention(cfg, c.handle, Q, O, c.workspace, dbg, stages)


def reference(case, code):
    if code == sa.SA_KV_FP16:
        cut = [slice(int(case.cu_lens[b]), int(case.cu_lens[b + 1])) for b in range(case.batch)]
        return np.stack([ora.sdpa_fp16(case.Q[b], case.K[s], case.V[s]) if s.stop > s.start else np.zeros(case.Q[b].shape) for b, s in enumerate(cut)]), None
    F = 0 if code == sa.SA_INT8 else 6 + code
    ref = ora.decode_attention(case.Q, case.K, case.V, case.cu_lens, code, F, hadamard=case.hadamard, want_scores=True, n_threads=8)
    return ref["O"], ref["A"]


@pytest.mark.parametrize("d,Hq,Hkv,code,dense,rot,lens,room", SHAPES)
def test_units_of_every_size_against_the_oracle(d, Hq, Hkv, code, dense, rot, lens, room):
    """Scores exact, outputs within 1e-3, the same bits whatever the workspace held before, and the two-launch form."""
    import torch
    sa_build.build()
    case = synth.make_case("stream", lens, Hq, Hkv, d, 0 if code == sa.SA_KV_FP16 else code, nibble=dense, hadamard=rot, outliers=True, seed=8100 + d + Hq + code)
    cfg = sa.make_config(d, Hq, Hkv, code, nibble=dense, hadamard=rot)
    c = wide_cache(cfg, lens, room)
    c.fill(up(case.K), up(case.V), case.cu_lens)
    Q, (want, scores) = up(case.Q), reference(case, code)
    first = None
    for contents in ("ones", "zeros", "random", "as left"):
        if contents == "zeros":
            c.workspace.zero_()
        elif contents == "random":
            c.workspace.copy_(torch.randint(0, 256, c.workspace.shape, generator=torch.Generator().manual_seed(3), dtype=torch.uint8))
        O = torch.full((len(lens), Hq, d), float("nan"), device="cuda")
        dbg = torch.full((len(lens), Hq, room), -7, dtype=torch.int32, device="cuda") if scores is not None and first is None else None
        attend(cfg, c, Q, O, dbg)
        torch.cuda.synchronize()
        assert marks(c.workspace) > 0 or len(lens) == 37      # units across blocks were merged in the kernel (37 x 4: one to a block)
        if first is None:
            first = O
            assert np.max(np.abs(O.cpu().numpy() - want)) <= 1e-3
            for b, n in enumerate(lens):
                if dbg is not None:
                    assert np.array_equal(dbg[b, :, :n].cpu().numpy().astype(np.int64), scores[b][:, :n]) and bool((dbg[b, :, n:] == -7).all())
        assert torch.equal(O, first), contents
    O = torch.full_like(first, float("nan"))
    attend(cfg, c, Q, O, stages=1)
    attend(cfg, c, Q, O, stages=2)
    # the same partials added in another order: FP32 sums of at most 148 terms, each within 2^-24 of a sum of magnitude below 8
    assert float((O - first).abs().max()) <= 148 * 8 * 2.0 ** -24


@pytest.mark.parametrize("d,Hq,Hkv,code,dense,rot,lens,room", [SHAPES[i] for i in (0, 1, 7, 10)])
def test_steps_equal_append_and_decode_bit_for_bit(d, Hq, Hkv, code, dense, rot, lens, room):
    """Several steps, as calls and replayed from a graph: bytes, lengths and outputs of sa_append_kv and a decode call; one sequence
    has no page for its token."""
    import torch
    sa_build.build()
    lens, n = np.asarray(lens), 3
    full = synth.make_case("stream", lens + n, Hq, Hkv, d, 0 if code == sa.SA_KV_FP16 else code, nibble=dense, hadamard=rot, seed=8200 + d)
    cfg = sa.make_config(d, Hq, Hkv, code, nibble=dense, hadamard=rot)
    old = np.concatenate([np.arange(full.cu_lens[b], full.cu_lens[b] + lens[b]) for b in range(len(lens))]).astype(np.int64)
    two = [wide_cache(cfg, lens, room, extra=n) for _ in range(2)]
    full_page = int(np.flatnonzero(lens == 64)[0])
    for c in two:
        c.fill(up(full.K[old]), up(full.V[old]), np.concatenate([[0], np.cumsum(lens)]))
        c.page_table[full_page, 1:] = -1
    ref, step = two
    lens0 = step.seq_lens.clone()
    Q = up(full.Q)
    new = [np.array([full.cu_lens[b] + lens[b] + i for b in range(len(lens))]) for i in range(n)]
    Kn, Vn = [up(full.K[x]) for x in new], [up(full.V[x]) for x in new]
    O = [[torch.full((len(lens), Hq, d), float("nan"), device="cuda") for _ in range(n)] for _ in range(2)]
    for i in range(n):
        sa.append_kv(cfg, ref.handle, Kn[i], Vn[i], True)
        attend(cfg, ref, Q, O[0][i])

    def steps():
        for i in range(n):
            sa.decode_step(cfg, step.handle, Q, Kn[i], Vn[i], O[1][i], step.workspace)

    steps()
    torch.cuda.synchronize()
    assert marks(step.workspace) > 0
    want_lens = lens + n
    want_lens[full_page] = 64
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        step.seq_lens.copy_(lens0)
        steps()
    for replay in range(2):
        assert step.seq_lens.cpu().numpy().tolist() == want_lens.tolist() == ref.seq_lens.cpu().numpy().tolist()
        assert all(torch.equal(a, b) for a, b in zip(*O)) and torch.equal(ref.pages, step.pages)
        for o in O[1]:
            o.fill_(float("nan"))
        graph.replay()
        torch.cuda.synchronize()


def test_lengths_rewritten_by_the_kernel_in_front_and_a_copy_that_never_comes():
    """The cut follows the lengths in force (those that the prologue saw may be others); a lost copy marks its rows and the call ends."""
    import torch
    sa_build.build()
    lens = [900, 64, 0, 2000, 33, 500, 70, 1] * 2
    case = synth.make_case("stream", lens, 32, 4, 64, 4, seed=8300)
    cfg = sa.make_config(64, 32, 4, sa.SA_POTM4)
    c = wide_cache(cfg, lens, 16384)
    c.fill(up(case.K), up(case.V), case.cu_lens)
    Q, orders = up(case.Q), [lens, [min(n, 40) for n in lens], [n // 2 for n in lens]]
    lens_dev = [torch.tensor(o, dtype=torch.int32, device="cuda") for o in orders]
    outs = [torch.full((16, 32, 64), float("nan"), device="cuda") for _ in range(9)]
    for i, O in enumerate(outs):                               # nothing synchronises inside this loop
        c.seq_lens.copy_(lens_dev[i % 3])
        attend(cfg, c, Q, O)
    torch.cuda.synchronize()
    for j, order in enumerate(orders):
        rows = np.concatenate([np.arange(case.cu_lens[b], case.cu_lens[b] + n) for b, n in enumerate(order)])
        want = ora.decode_attention(case.Q, case.K[rows], case.V[rows], np.concatenate([[0], np.cumsum(order)]), 4, 10, n_threads=8)["O"]
        for O in outs[j::3]:
            assert np.max(np.abs(O.cpu().numpy() - want)) <= 1e-3
    c.seq_lens.copy_(lens_dev[0])
    O = torch.zeros((16, 32, 64), device="cuda")
    sa.debug_decode_lost_copy(cfg, c.handle, Q, O, c.workspace, 3, 1, 20)
    torch.cuda.synchronize()
    assert bool(torch.isnan(O[3, 8:16]).all()) and bool(torch.isfinite(O[:, :8]).all())
    attend(cfg, c, Q, O)                                       # and the next call is an ordinary one
    assert torch.equal(O, outs[0])


@pytest.mark.parametrize("byte", range(8))
def test_words_at_rest_of_which_one_byte_was_overwritten(byte):
    """The counting words that a call leaves are memory like any other: a byte written into each changes no later call."""
    import torch
    sa_build.build()
    d, Hq, Hkv, code, dense, rot, lens, room = SHAPES[0]
    case = synth.make_case("stream", lens, Hq, Hkv, d, code, seed=8500)
    cfg = sa.make_config(d, Hq, Hkv, code)
    c = wide_cache(cfg, lens, room, extra=1)
    c.fill(up(case.K), up(case.V), case.cu_lens)
    Q, K, V = up(case.Q), up(case.K[:len(lens)]), up(case.V[:len(lens)])
    lens0, outs = c.seq_lens.clone(), []
    for call in range(4):
        if call:
            words = c.workspace[:len(c.workspace) // 8 * 8].view(torch.int64)
            rest = (words >> 24) == MARK
            assert int(rest.sum()) > 1
            words[rest] ^= 5 << (8 * byte)
        c.seq_lens.copy_(lens0)
        O = torch.full((len(lens), Hq, d), float("nan"), device="cuda")
        sa.decode_step(cfg, c.handle, Q, K, V, O, c.workspace)
        torch.cuda.synchronize()
        outs.append(O)
        assert torch.equal(c.seq_lens, lens0 + 1)
        assert torch.equal(O, outs[0])


@pytest.mark.parametrize("d,Hq,Hkv,code,batch", [(64, 32, 4, sa.SA_POTM4, 32), (64, 32, 4, sa.SA_INT8, 16), (128, 32, 8, sa.SA_POTM4, 8)])
def test_sums_over_long_stretches_against_64_bits(d, Hq, Hkv, code, batch):
    """Values of mean 1, whose sums grow with every tile: up to 55 tiles a warp.  The matrix unit cuts its sums off, by up to 2^-23;
    four of them make a tile: 4.8e-7.  Weights of 21 bits (2.4e-7) and the tiles' sums, rounded to nearest
    (sqrt(55) 2^-24, 4.4e-7), are added: 1.2e-6 of the largest output at most, 1e-6 in the mean square."""
    import torch
    sa_build.build()
    n = 32768
    gen = torch.Generator(device="cuda").manual_seed(8600 + d + code)
    cfg = sa.make_config(d, Hq, Hkv, code)
    c = sa.PagedCache(cfg, [n] * batch, "cuda", permutation=synth.page_permutation(batch * n // 64, 3))
    K = torch.randn((batch * n, Hkv, d), generator=gen, device="cuda").half()
    V = (torch.randn((batch * n, Hkv, d), generator=gen, device="cuda") + 1).half()
    c.fill(K, V, np.arange(batch + 1) * n)
    del K, V
    Q = torch.randn((batch, Hq, d), generator=gen, device="cuda").half()
    O = torch.full((batch, Hq, d), float("nan"), device="cuda")
    c.workspace.fill_(255)
    attend(cfg, c, Q, O)
    assert marks(c.workspace) > 0
    q_hat, delta = torch.zeros((batch, Hq, d), dtype=torch.int8, device="cuda"), torch.zeros((batch, Hq), device="cuda")
    sa.quantise_query(cfg, Q, q_hat, delta)
    q = (q_hat.double() * delta.double()[..., None])[0]
    codes, v_hat = [torch.zeros((n, Hkv, d), dtype=t, device="cuda") for t in (torch.uint8, torch.int8)]
    scales, g = [torch.zeros((n, Hkv), dtype=t, device="cuda") for t in (torch.float16, torch.int8)]
    sa.debug_unpack(cfg, c.handle, 0, n, codes, scales, v_hat, g)
    if code == sa.SA_INT8:
        keys = codes.view(torch.int8).double() / 127
    else:
        keys = torch.where(codes >= 128, -1.0, 1.0).double() * (1 + (codes & 15).double() / 16) * torch.exp2(-((codes >> 4) & 7).double())
        keys[((codes >> 4) & 7) == 7] = 0
    keys, values, G = keys * scales.double()[..., None], v_hat.double() * torch.exp2(-g.double())[..., None], Hq // Hkv
    want = torch.cat([torch.softmax(q[h * G:(h + 1) * G] @ keys[:, h].T / d ** 0.5, -1) @ values[:, h] for h in range(Hkv)])
    off = O[0].double() - want
    assert float(off.abs().max() / want.abs().max()) <= 1.2e-6 and float(off.norm() / want.norm()) <= 1e-6


# equal lengths, 64 tokens a page, room for `room`: units (sequences x KV heads) in 2 and 4 even parts, with tiles to spare and without,
# fewer tiles than parts, one to a block, whole ones one after another, and so many tiles that the cut takes no notice of units
EQUAL = [(64, 16, 2, sa.SA_POTM4, False, 37, [1, 33, 2000, 4000], 32768), (64, 8, 1, sa.SA_POT4, True, 37, [31, 100, 4000], 32768),
         (64, 32, 4, sa.SA_POT4, False, 37, [0, 65, 777], 65536), (64, 32, 4, sa.SA_POTM4, False, 48, [96, 600], 16384),
         (128, 16, 16, sa.SA_POTM2, True, 16, [64, 500, 1500], 8192), (128, 32, 8, sa.SA_POTM4, False, 8, [200, 900, 3000], 8192),
         (64, 32, 4, sa.SA_KV_FP16, False, 32, [40, 700], 8192), (64, 8, 1, sa.SA_INT8, False, 100, [32, 1300], 16384)]


@pytest.mark.parametrize("d,Hq,Hkv,code,dense,batch,tokens,room", EQUAL)
def test_units_of_equal_lengths_against_the_oracle(d, Hq, Hkv, code, dense, batch, tokens, room):
    """Every sequence has the same keys and queries, so all outputs are those of the first, whose are the oracle's."""
    import torch
    sa_build.build()
    cfg = sa.make_config(d, Hq, Hkv, code, nibble=dense)
    for n in tokens:
        case = synth.make_case("equal", [n], Hq, Hkv, d, 0 if code == sa.SA_KV_FP16 else code, nibble=dense, outliers=True, seed=8700 + n)
        want, scores = reference(case, code)
        c = wide_cache(cfg, [n] * batch, room)
        c.fill(*[up(np.concatenate([x] * batch)) for x in (case.K, case.V)], np.arange(batch + 1) * n)
        Q = up(np.concatenate([case.Q] * batch))
        dbg = torch.full((batch, Hq, room), -7, dtype=torch.int32, device="cuda") if scores is not None else None
        for call in range(2):
            O = torch.full((batch, Hq, d), float("nan"), device="cuda")
            attend(cfg, c, Q, O, dbg if call else None)
            torch.cuda.synchronize()
            assert np.max(np.abs(O.cpu().numpy() - want[:1])) <= 1e-3, n
        if dbg is not None:
            assert np.array_equal(dbg[:, :, :n].cpu().numpy(), np.broadcast_to(scores[0][None, :, :n], (batch, Hq, n))) and bool((dbg[:, :, n:] == -7).all())
        attend(cfg, c, Q, O.fill_(float("nan")), stages=1)
        attend(cfg, c, Q, O, stages=2)
        assert np.max(np.abs(O.cpu().numpy() - want[:1])) <= 1e-3, n
