"""The span that kb_search_span reports: the shapes kb_search launches (a host function: no GPU needed)."""
import pytest

from paper_1901_02492_gb300 import binding as kb

R, P = kb.KB_RESCORE_FP64, kb.KB_PRUNE


@pytest.mark.parametrize("storage,variant,V,topk,flags,span", [
    ("f32", 0, 1024, 8, 0, 64), ("f32", 0, 1024, 16, 0, 64), ("f32", 0, 1024, 8, P, 64), ("f32", 0, 640, 8, R, 64),
    ("f32", 1, 64, 8, 0, 128), ("f32", 2, 64, 8, 0, 64), ("f32", 3, 64, 8, 0, 128), ("f32", 4, 64, 8, 0, 64),
    # 16-bit value lists: one pair of pixels per lane; pruned short ones two
    ("bf16", 0, 1024, 8, 0, 64), ("f16", 0, 1024, 1, 0, 64), ("bf16", 0, 1024, 9, 0, 64), ("bf16", 0, 1024, 8, P, 128),
    ("bf16", 0, 1024, 9, P, 64),
    # key lists (up to 16 candidates, 4096 velocities): two pairs; longer lists and more velocities: value lists
    ("bf16", 0, 640, 4, R, 128), ("bf16", 0, 640, 8, R, 128), ("bf16", 0, 4096, 10, R, 128), ("bf16", 0, 4097, 10, R, 64),
    ("bf16", 0, 640, 12, R, 64), ("f16", 0, 640, 12, R, 128), ("bf16", 0, 640, 8, R | P, 64), ("bf16", 0, 640, 4, R | P, 128),
    ("bf16", 1, 64, 8, 0, 128), ("bf16", 2, 64, 8, R, 64), ("f16", 3, 64, 16, 0, 128), ("f16", 4, 64, 16, 0, 64),
    ("f32", 5, 64, 8, 0, 64), ("bf16", 8, 64, 8, 0, 128)])
def test_span_of_the_launched_shape(storage, variant, V, topk, flags, span):
    assert kb.search_span(storage, variant, V, topk, flags) == span


@pytest.mark.parametrize("args", [("f32", 9, 8, 8, 0), ("f32", 0, 0, 8, 0), ("f32", 0, 8, 17, 0), ("f32", 0, 8, 8, 64)])
def test_span_refuses_what_a_search_refuses(args):
    with pytest.raises(kb.KBError):
        kb.search_span(*args)
