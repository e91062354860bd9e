"""The host's split plan (no GPU): what is kept per shape must not leak between configurations."""
from paper_2609_09208_b200 import binding as sa


def test_workspace_size_does_not_depend_on_what_was_asked_before():
    """Configurations that share the shape but not the kernel do not share the plan, in whichever order they ask."""
    def sizes(order):
        return {c: [sa.workspace_bytes(sa.make_config(64, 32, 4, c[0], add_on_alu=c[1]), b, p) for b in (1, 3, 32) for p in (40, 512)]
                for c in order}
    configs = [(sa.SA_POTM4, False), (sa.SA_POTM1, True), (sa.SA_INT8, False), (sa.SA_POTM1, False), (sa.SA_KV_FP16, False), (sa.SA_POTM4, True)]
    assert sizes(configs) == sizes(configs[::-1])


def test_shift_by_multiply_has_the_shift_kernels_plan():
    """SA_FLAG_SHIFT_BY_MULTIPLY selects kernels of its own, with the shape of the shift-and-add kernels, and not the default."""
    for code, nibble in [(sa.SA_POTM1, False), (sa.SA_POTM1, True), (sa.SA_POTM2, True), (sa.SA_POTM4, False)]:
        size = lambda **flags: [sa.workspace_bytes(sa.make_config(d, 32, 4, code, nibble=nibble, **flags), b, p)
                                for d in (64, 128) for b in (1, 3, 7, 32) for p in (20, 40, 100, 512, 700)]
        assert size(shift_by_multiply=True) == size(add_on_alu=True) != size()


def test_the_shapes_of_the_stream_tests_go_to_the_kernel_of_one_block_per_sm():
    """Its workspace (148 SMs: a slot per block and unit boundary, words, plan, in whole splits) is another one than the other kernel's."""
    from test_gpu_stream import EQUAL, SHAPES
    shapes = [(d, Hq, Hkv, code, dense, len(lens), room) for d, Hq, Hkv, code, dense, _, lens, room in SHAPES]
    for d, Hq, Hkv, code, dense, batch, room in shapes + [x[:6] + x[7:] for x in EQUAL]:
        gt = next(c for c in (8, 4, 2, 1) if Hq // Hkv % c == 0)
        units, split = batch * Hkv * (Hq // Hkv // gt), batch * Hq * (d + 2) * 4
        need = (148 + units) * gt * (d + 2) * 4 + (units + 1) * 8 + units * 8
        size = sa.workspace_bytes(sa.make_config(d, Hq, Hkv, code, nibble=dense), batch, room // 64) - (batch * 8 + 15) // 16 * 16
        # (37 sequences of PoT-M1 with room for 8192 tokens stay with the other kernel)
        assert (size == -(-need // split) * split) == ((batch, room) != (37, 8192)), (d, Hq, Hkv, code, batch, room)


def test_binary16_units_that_fill_the_machine_once_stay_unsplit():
    """64 sequences of 4 KV heads, 256 units on 296 slots: one split and no workspace of the kernel of one block per SM."""
    cfg = sa.make_config(64, 32, 4, sa.SA_KV_FP16)
    for tokens in (4096, 8192):
        assert sa.workspace_bytes(cfg, 64, tokens // 64) == 64 * 32 * 66 * 4 + 64 * 8
