"""Sizes that just fit the forward's scratch: the workspace-free forward takes them (its array holds 32 MiB)."""
import pytest

import paper_2408_15766_b200 as hass


# 1774 to 1776 (row tile, lane) slots: with 512 bytes more for each they would need up to 33.0 MiB
@pytest.mark.parametrize("N,V", [(3072, 132352), (6528, 123136), (7552, 104192)])
def test_sizes_that_just_fit_are_taken(N, V):
    assert hass.topk_distill_fwd_static_scratch_bytes(N, 64, V, 16) <= 32 << 20
