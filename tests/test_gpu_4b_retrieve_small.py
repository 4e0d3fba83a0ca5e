"""Retrieval at the edges of what its variants take: candidate counts around
the insertion limit of the small-batch kernel, corpora of a few tiles for
k <= 32 and beyond, equal scores everywhere, and merges of few rows (Section
4.1: the k best chunks per query, ties to the lower index)."""
import numpy as np
import pytest
import torch

import paper_2607_22578_gb300 as hs
import synth
from hs_testutil import bf16_f64, graph_us, to_dev

pytestmark = pytest.mark.gpu


def check(Q, C, k):
    s, i = hs.hs_retrieve_topk(to_dev(Q).view(torch.bfloat16), to_dev(C).view(torch.bfloat16), k)
    hs.hs_get_device_error()
    full = bf16_f64(Q) @ bf16_f64(C).T
    order = np.lexsort((np.broadcast_to(np.arange(len(C)), full.shape), -full))[:, :k]
    want = np.take_along_axis(full, order, 1)
    s, i = s.cpu().numpy(), i.cpu().numpy()
    assert np.abs(s - want).max() < 1e-3
    assert np.abs(np.take_along_axis(full, i.astype(np.int64), 1) - want).max() < 1e-3
    assert all(len(set(r)) == k for r in i.tolist())
    return s, i, order


@pytest.mark.parametrize("k", [1, 3, 4, 10, 16, 17, 32])
@pytest.mark.parametrize("nq,N", [(1, 127), (5, 129), (16, 5000), (17, 300), (64, 4096),
                                  (152, 2000), (153, 2000), (300, 777)])
def test_register_lists_on_small_corpora(nq, N, k):
    check(synth.unit_rows(nq, 72, nq + k), synth.unit_rows(N, 72, N), k)


@pytest.mark.parametrize("nq,N,k", [(3, 40, 33), (20, 256, 64), (5, 300, 64), (130, 1000, 100),
                                    (260, 2000, 200), (40, 16000, 500), (9, 4096, 1024)])
def test_large_k_on_few_tiles(nq, N, k):
    check(synth.unit_rows(nq, 64, nq), synth.unit_rows(N, 64, N + k), k)


@pytest.mark.parametrize("k", [5, 32, 100])
def test_large_k_crowded_into_one_tile(k):
    """The top k of every query lies in one tile of the corpus: the lists of
    the optimistic pass are cut, and the blocks run the exact pass."""
    C = synth.unit_rows(3000, 64, 5)
    Q = np.tile(synth.unit_rows(1, 64, 6), (150, 1))
    near = bf16_f64(Q[:1]).astype(np.float32) + np.linspace(0.0, 0.3, 200)[:, None].astype(
        np.float32) * bf16_f64(C[:200]).astype(np.float32)
    near /= np.linalg.norm(near, axis=1, keepdims=True)
    C[520:720] = torch.from_numpy(near).to(torch.bfloat16).view(torch.int16).numpy().view(np.uint16)
    check(Q, C, k)


@pytest.mark.parametrize("nq", [1, 16, 17, 200])
@pytest.mark.parametrize("k", [4, 10, 32, 40])
def test_equal_scores_go_to_the_lowest_rows(nq, k):
    C = np.tile(synth.unit_rows(1, 64, 1), (1500, 1))
    s, i, order = check(np.tile(synth.unit_rows(1, 64, 2), (nq, 1)), C, k)
    assert (i == np.arange(k)).all() and (s == s[0, 0]).all()


@pytest.mark.parametrize("nq", [2, 40])
def test_scores_of_the_lowest_value_and_ascending_rows(nq):
    """Every row beats the ones before it, and zero rows (score 0) among
    negative ones: each tile replaces the whole list."""
    base = bf16_f64(synth.unit_rows(1, 64, 3))[0]
    scale = np.linspace(-1.0, -0.01, 2000)
    scale[::97] = 0.0
    rows = torch.from_numpy((scale[:, None] * base).astype(np.float32)).to(torch.bfloat16)
    C = rows.view(torch.int16).numpy().view(np.uint16)
    check(np.tile(synth.unit_rows(1, 64, 3), (nq, 1)), C, 10)


@pytest.mark.parametrize("d", [8, 64, 136, 768, 1024, 1032])
@pytest.mark.parametrize("nq", [17, 31, 33, 63, 64, 65])
def test_resident_queries(nq, d):
    """17 to 64 queries stay in shared memory (d <= 1024): widths around a
    64-dimension block, row counts around a 128-row tile, several tiles per CTA."""
    for N, k in ((127, 7), (129, 12), (385, 16), (25001, 32)):
        check(synth.unit_rows(nq, d, nq + N), synth.unit_rows(N, d, N), k)


def test_resident_queries_with_the_count_on_the_device():
    q, c = synth.unit_rows(64, 128, 1), synth.unit_rows(9000, 128, 2)
    Q, C = (to_dev(x).view(torch.bfloat16) for x in (q, c))
    Q[40:] = float("nan")                          # rows past the count are never selected from
    want_s, want_i = hs.hs_retrieve_topk(Q[:40].contiguous(), C, 10)
    for n in (0, 1, 39, 40):
        s = torch.full((64, 10), 7.0, device="cuda")
        i = torch.full((64, 10), 7, dtype=torch.int32, device="cuda")
        hs.hs_retrieve_topk_n(Q, torch.tensor([n], dtype=torch.int32, device="cuda"), C, 10,
                              out=(s, i))
        hs.hs_get_device_error()
        assert torch.equal(s[:n], want_s[:n]) and torch.equal(i[:n], want_i[:n])
        assert (s[n:] == 7.0).all() and (i[n:] == 7).all()


def test_resident_pipeline_wait_runs_out():
    """As the other kernels' waits: a stage that never fills ends in
    HS_ERR_TIMEOUT, and the next call is right."""
    q, c = synth.unit_rows(40, 256, 3), synth.unit_rows(30000, 256, 4)
    Q, C = (to_dev(x).view(torch.bfloat16) for x in (q, c))
    want = hs.hs_retrieve_topk(Q, C, 10)
    try:
        hs.hs_debug_retrieve_wait(1_000_000, 1)
        hs.hs_retrieve_topk(Q, C, 10)
        with pytest.raises(hs.HsError) as e:
            hs.hs_get_device_error()
        assert e.value.status == hs.HS_ERR_TIMEOUT
    finally:
        hs.hs_debug_retrieve_wait()
    got = hs.hs_retrieve_topk(Q, C, 10)
    hs.hs_get_device_error()
    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])


@pytest.mark.parametrize("crowd", [0, 14, 40])
@pytest.mark.parametrize("k", [17, 32, 50, 128, 129])
@pytest.mark.parametrize("nq", [3, 40, 600])
def test_lists_shorter_than_k(nq, k, crowd):
    """More than 16 results from lists of 12 to 32 slots: a query's best rows
    spread over the corpus, or 14 and 40 of them side by side, which cuts a
    list of the first pass, and of the second as well; only some query blocks
    have such a query."""
    C = synth.unit_rows(9000, 64, k)
    Q = synth.unit_rows(nq, 64, 6)
    if crowd:
        q = bf16_f64(Q[nq // 2:nq // 2 + 1])
        near = q + np.linspace(0.0, 0.3, crowd)[:, None] * bf16_f64(C[:crowd])
        near /= np.linalg.norm(near, axis=1, keepdims=True)
        bits = torch.from_numpy(near.astype(np.float32)).to(torch.bfloat16).view(torch.int16)
        C[4100:4100 + crowd] = bits.numpy().view(np.uint16)
    check(Q, C, k)


@pytest.mark.parametrize("k", [24, 60])
@pytest.mark.parametrize("n_live", [1, 150, 400])
def test_lists_shorter_than_k_with_fanout(n_live, k):
    """The same through a device count and a fan-out map, where several rows
    hand the same cut query on: every row gets its query's result."""
    rng = np.random.default_rng(k)
    C = synth.unit_rows(9000, 64, k)
    Q = synth.unit_rows(400, 64, 6)
    for j, q in enumerate(range(0, n_live, 7)):
        near = bf16_f64(Q[q:q + 1]) + np.linspace(0.0, 0.3, 20)[:, None] * bf16_f64(C[:20])
        near /= np.linalg.norm(near, axis=1, keepdims=True)
        bits = torch.from_numpy(near.astype(np.float32)).to(torch.bfloat16).view(torch.int16)
        C[130 * j + 100:130 * j + 120] = bits.numpy().view(np.uint16)
    inv = rng.integers(0, n_live, size=1000).astype(np.int32)
    dq, dc = to_dev(Q).view(torch.bfloat16), to_dev(C).view(torch.bfloat16)
    s, i = hs.hs_retrieve_topk_fanout(dq, to_dev(np.array([n_live], np.int32)), to_dev(inv), dc, k)
    hs.hs_get_device_error()
    full = bf16_f64(Q[:n_live]) @ bf16_f64(C).T
    want = -np.sort(-full, axis=1)[:, :k][inv]
    s, i = s.cpu().numpy(), i.cpu().numpy().astype(np.int64)
    assert np.abs(s - want).max() < 1e-3
    assert np.abs(np.take_along_axis(full[inv], i, 1) - want).max() < 1e-3


def test_small_batch_merge_with_few_sms_free():
    """8 queries over 19,000 rows, whose 150 CTAs leave 2 SMs free: no dearer than over
    20,480 (1.4 times with the merge's blocks launched early, all onto those two)."""
    us = []
    for n in (19000, 20480):
        q, c = (to_dev(synth.unit_rows(m, 128, m)).view(torch.bfloat16) for m in (8, n))
        ws = torch.empty(hs.hs_retrieve_topk_workspace(8, n, 128, 10), dtype=torch.uint8,
                         device="cuda")
        out = (torch.empty((8, 10), device="cuda"),
               torch.empty((8, 10), dtype=torch.int32, device="cuda"))
        us.append(graph_us(lambda: hs.hs_retrieve_topk(q, c, 10, workspace=ws, out=out)))
    hs.hs_get_device_error()
    assert us[0] < 1.15 * us[1], us
