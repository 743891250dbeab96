"""The tensors the binding makes for a routing call (host side, no GPU): each one an allocation of its own."""
import itertools

import pytest
import torch

from paper_2607_19438_b200 import binding


@pytest.mark.parametrize("M,E,k", [(5, 7, 1), (1, 1, 1), (4, 128, 8), (3, 5, 3), (0, 4, 2)])
def test_outputs_are_aligned_and_share_no_storage(M, E, k):
    o = binding._route_outputs(torch.zeros((M, E)), k, torch.zeros((M, 24), dtype=torch.bfloat16), None)
    shapes = dict(topk_idx=(M, k), topk_w=(M, k), counts=(E,), offsets=(E + 1,), row_pair=(M * k,), pair_row=(M * k,), Xperm=(M * k, 24))
    assert {n: tuple(t.shape) for n, t in o.items()} == shapes
    assert {n: t.dtype for n, t in o.items()} == {n: torch.int32 for n in shapes} | dict(topk_w=torch.float32, Xperm=torch.bfloat16)
    assert all(t.data_ptr() % 16 == 0 and t.is_contiguous() and t.storage_offset() == 0 for t in o.values())
    for a, b in itertools.combinations((t for t in o.values() if t.numel()), 2):
        assert a.untyped_storage().data_ptr() != b.untyped_storage().data_ptr()


def test_an_output_changed_in_place_leaves_the_others_usable_in_a_backward_pass():
    logits = torch.randn((4, 8), requires_grad=True)
    o = binding._route_outputs(logits.detach(), 2, None, None)
    o["topk_idx"].zero_()
    o["topk_w"].fill_(1.0)
    picked = torch.nn.functional.embedding(o["topk_idx"], logits.T).sum()       # keeps topk_idx for its backward
    o["topk_w"].mul_(2.5)                                                       # a routing scale, applied in place
    picked.backward()
    assert float(logits.grad.sum()) == 32.0
