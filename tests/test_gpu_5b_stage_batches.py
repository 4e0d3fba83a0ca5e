"""One stage serving batches of many sizes in turn (Section 4.1): every size
gives what a stage of its own gives, with and without the result cache, and a
returned tensor is the caller's to reshape."""
import pytest
import torch

import paper_2607_22578_gb300 as hs
import synth
from hs_testutil import to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cache", [0, 4096])
def test_many_batch_sizes_through_one_stage(cache):
    corpus = to_dev(synth.unit_rows(2000, 64, 1)).view(torch.bfloat16)
    queries = to_dev(synth.unit_rows(300, 64, 2)).view(torch.bfloat16)
    queries[100:150] = queries[:50]
    stage = hs.EmbedRetrieveStage(corpus, 5, 300, cache_capacity=cache)
    whole_s, whole_i, nu = stage.retrieve(queries)
    want_s, want_i = whole_s.clone(), whole_i.clone()
    assert int(nu.item()) == 250
    for n in list(range(1, 300, 7)) + [256, 257, 300, 1, 256]:
        s, i, nu = stage.retrieve(queries[:n])
        assert torch.equal(s, want_s[:n]) and torch.equal(i, want_i[:n])
        assert int(nu.item()) == n - max(0, min(n, 150) - 100)
        s.unsqueeze_(0), i.t_()                     # shapes of this call's tensors only
    hs.hs_get_device_error()
