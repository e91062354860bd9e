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
