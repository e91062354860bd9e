"""The library's exact-arithmetic functions, compiled for the host, against the CPU oracle.

The key-element encoder, the value exponent and the packed-shift and table score datapaths are plain
integer code that nvcc also compiles for the host; this checks them exhaustively / on random
inputs without a GPU.  (The same functions run on the device in the -m gpu parity tests.)"""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

from oracle import sa_oracle as ora

HERE = os.path.dirname(os.path.abspath(__file__))
SRC = os.path.join(HERE, "host_harness.cu")
LIB = os.path.join(HERE, "_build", "libhh.so")
CSRC = os.path.join(HERE, "..", "paper_2609_09208_b200", "csrc")


@pytest.fixture(scope="module")
def hh():
    os.makedirs(os.path.dirname(LIB), exist_ok=True)
    deps = [SRC] + [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith(".cuh")]
    if not os.path.exists(LIB) or any(os.path.getmtime(d) > os.path.getmtime(LIB) for d in deps):
        subprocess.check_call(["/usr/local/cuda/bin/nvcc", "-gencode", "arch=compute_100a,code=sm_100a", "-std=c++17", "-O2", "-shared",
                               "-Xcompiler", "-fPIC", "-o", LIB, SRC])
    lib = C.CDLL(LIB)
    return lib


SCALES = [0x3C00, 0x7BFF, 0x3A66, 0x0400, 0x01F3, 0x4D2B, 0x0001, 0x2E66]


@pytest.mark.parametrize("k", [0, 1, 2, 4])
@pytest.mark.parametrize("s_bits", SCALES)
def test_encode_element_exhaustive_vs_oracle(hh, k, s_bits):
    mags = np.arange(0, s_bits + 1, dtype=np.uint16)
    vals = (mags | ((np.arange(len(mags)) % 2).astype(np.uint16) << 15)).astype(np.uint16)
    got = np.empty(len(vals), dtype=np.uint8)
    hh.hh_encode_many(C.c_int(k), vals.ctypes.data_as(C.c_void_p), C.c_int64(len(vals)), C.c_uint(s_bits),
                      got.ctypes.data_as(C.c_void_p))
    d = 64
    n_vec = (len(vals) + d - 2) // (d - 1)
    K = np.zeros((n_vec, d), dtype=np.uint16)
    K[:, 0] = s_bits
    flat = np.zeros(n_vec * (d - 1), dtype=np.uint16)
    flat[: len(vals)] = vals
    K[:, 1:] = flat.reshape(n_vec, d - 1)
    want = ora.encode_keys(K, k)[0][:, 1:].reshape(-1)[: len(vals)]
    assert np.array_equal(got, want)


def test_value_exponent_all_magnitudes(hh):
    mags = np.arange(0, 0x7C00, dtype=np.uint16)          # every finite binary16 magnitude
    V = np.zeros((len(mags), 64), dtype=np.uint16)
    V[:, 5] = mags
    _, g = ora.quantise_value(V)
    got = np.array([hh.hh_value_exponent(C.c_uint(int(m))) for m in mags], dtype=np.int8)
    assert np.array_equal(got, g)


@pytest.mark.parametrize("k", [0, 1, 2, 4])
@pytest.mark.parametrize("d", [64, 128])
def test_score_datapaths_equal_oracle_scores(hh, k, d):
    """Eight queries (two per 32-bit register) against one key through the kernel's word decoders
    and packed accumulators, including the cases that stress the 16-bit halves: every term
    negative at the largest shift, extreme queries, zero codes with and without a sign bit."""
    rng = np.random.default_rng(100 + k + d)
    out = np.zeros(8, dtype=np.int32)
    for trial in range(300):
        e = rng.integers(0, 8, d)
        j = rng.integers(0, 1 << k, d)
        sgn = rng.integers(0, 2, d)
        if trial % 7 == 1:
            e[:] = 0                                # largest shift everywhere
        if trial % 7 == 2:
            sgn[:] = 1
        if trial % 7 == 3:
            j[:] = (1 << k) - 1
        codes = ((sgn << 7) | (e << 4) | (j << (4 - k))).astype(np.uint8)
        if trial % 3 == 0:
            codes[e == 7] = 0x70                    # canonical zeros (otherwise: zero codes keep their sign bit)
        else:
            codes[e == 7] &= 0xF0                   # a zero code has no mantissa bits
        q = rng.integers(-127, 128, (8, d)).astype(np.int8)
        if trial % 5 == 1:
            q[:] = 127
        if trial % 5 == 2:
            q[::2] = -127
            q[1::2] = 127
        if trial % 5 == 3:
            q[:] = -127
        want, ov = ora.scores(q, codes[None, None, :], k, 6 + k)
        assert ov == 0
        hh.hh_score8(C.c_int(k), codes.ctypes.data_as(C.c_void_p), q.ctypes.data_as(C.c_void_p), C.c_int(d),
                     C.c_int(0), out.ctypes.data_as(C.c_void_p))
        assert np.array_equal(out.astype(np.int64), want[:, 0]), (trial, out, want[:, 0])
        if k == 0:
            hh.hh_score8(C.c_int(0), codes.ctypes.data_as(C.c_void_p), q.ctypes.data_as(C.c_void_p), C.c_int(d),
                         C.c_int(1), out.ctypes.data_as(C.c_void_p))
            assert np.array_equal(out.astype(np.int64), want[:, 0]), ("nibble", trial)
        else:
            # the table datapath of the mantissa codes gives the same integers
            hh.hh_score8_table(C.c_int(k), codes.ctypes.data_as(C.c_void_p), q.ctypes.data_as(C.c_void_p), C.c_int(d),
                               out.ctypes.data_as(C.c_void_p))
            assert np.array_equal(out.astype(np.int64), want[:, 0]), ("table", trial, out, want[:, 0])
            if k in (1, 2):
                # ... and so does the dense planar container (nibbles + mantissa bit planes)
                hh.hh_score8_planar(C.c_int(k), codes.ctypes.data_as(C.c_void_p), q.ctypes.data_as(C.c_void_p), C.c_int(d),
                                    out.ctypes.data_as(C.c_void_p))
                assert np.array_equal(out.astype(np.int64), want[:, 0]), ("planar", trial, out, want[:, 0])
        # the non-default kernels that run the shifts on the integer multiplier: the same integers again
        for path in (() if k == 0 else (0, 1) if k in (1, 2) else (0,)):
            hh.hh_score8_mul(C.c_int(k), codes.ctypes.data_as(C.c_void_p), q.ctypes.data_as(C.c_void_p), C.c_int(d),
                             C.c_int(path), out.ctypes.data_as(C.c_void_p))
            assert np.array_equal(out.astype(np.int64), want[:, 0]), ("shift by multiply", path, trial, out, want[:, 0])
        # the non-default kernels without any multiply-add (sign flip and add as logic and add instructions)
        for path in ((0, 1) if k in (0, 1, 2) else (0,)):
            hh.hh_score8_alu(C.c_int(k), codes.ctypes.data_as(C.c_void_p), q.ctypes.data_as(C.c_void_p), C.c_int(d),
                             C.c_int(path), out.ctypes.data_as(C.c_void_p))
            assert np.array_equal(out.astype(np.int64), want[:, 0]), ("adds on the ALU pipe", path, trial, out, want[:, 0])


@pytest.mark.parametrize("devs,fails,calls", [
    ([0, 0, 1, 0, 1, 1], [0] * 6, 2),                    # once on each device, not once in the process
    ([0, 0, 0], [1, 0, 0], 2),                           # what was refused is asked for again
    ([63, 63, 64, 64, 70], [0] * 5, 4)])                 # beyond the table: each time
def test_kernel_attributes_are_set_once_per_device(hh, devs, fails, calls):
    n = len(devs)
    ok = (C.c_int * n)()
    assert hh.hh_once_per_device((C.c_int * n)(*devs), (C.c_int * n)(*fails), C.c_int(n), ok) == calls
    assert list(ok) == [1 - f for f in fails]


@pytest.mark.parametrize("shape,appends,want", [
    ((8, 4, 8, 8, 1), 1, 7), ((8, 4, 8, 8, 1), 0, 5),                      # a cluster of eight; nothing to count without an append
    ((1, 256, 8, 8, 65535), 1, 7), ((1, 256, 8, 4, 65535), 1, 4),          # 2^24 - 256 blocks are counted, twice as many are not
    ((1, 256, 1, 1, 65536), 1, 4), ((1, 256, 8, 4, 65535), 0, 5)])
def test_steps_of_one_launch_have_at_most_as_many_blocks_as_the_word_counts(hh, shape, appends, want):
    """settle_whole(splits, KV heads, group, queries per block, batch): one launch (1), counting word (2), cluster kept (4)."""
    assert hh.hh_settle_whole(*[C.c_int(x) for x in shape], C.c_int(appends)) == want


REST = 0x7fa5c3d296 << 24                            # a counting word without arrivals


def arrive(hh, contents, blocks, calls, late=False):
    hh.hh_arrive.restype = C.c_uint64
    last = np.zeros(calls, dtype=np.uint8)
    word = hh.hh_arrive(C.c_uint64(contents), C.c_int(blocks), C.c_int(calls), C.c_int(late), last.ctypes.data_as(C.c_void_p))
    return word, np.flatnonzero(last).tolist()


@pytest.mark.parametrize("blocks", [1, 2, 5, 148])
def test_counting_word_of_any_contents_names_the_last_block_and_ends_at_rest(hh, blocks):
    """Every single byte of a word at rest changed, its halves overwritten, and words near it."""
    words = [REST, 0, 2**64 - 1, 0xFFFFFFFF, REST - 1, REST - 2**32, REST - 1 - 2**32, REST + 1, REST + 2**32, (REST >> 32) << 32, REST & 0xFFFFFFFF]
    words += [REST ^ (x << (8 * byte)) for byte in range(8) for x in (1, 2, 5, 0x80, 0xFF)]
    words += [int(x) for x in np.random.default_rng(1).integers(0, 2**64, 200, dtype=np.uint64)]
    for w in words:
        assert arrive(hh, w, blocks, blocks) == (REST, [blocks - 1]), hex(w)
        assert arrive(hh, w, blocks, 3 * blocks) == (REST, [blocks - 1, 2 * blocks - 1, 3 * blocks - 1]), hex(w)


@pytest.mark.parametrize("blocks", [2, 5, 148])
def test_counting_word_is_at_rest_again_after_calls_that_overlapped(hh, blocks):
    assert arrive(hh, REST, blocks, 3 * blocks, late=True) == (REST, [blocks - 1, 2 * blocks - 1, 3 * blocks - 1])
