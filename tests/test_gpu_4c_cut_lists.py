"""Retrieval of more than 16 results where a query's best rows are neighbours
in the corpus, as the chunks of a document are (Section 4.1): the first pass's
short lists are cut, run again over their own rows, and cut again or not."""
import numpy as np
import pytest
import torch

import paper_2607_22578_gb300 as hs
import synth
from hs_testutil import bf16_f64, graph_us, to_dev

pytestmark = pytest.mark.gpu


def bits(x):
    return torch.from_numpy(np.asarray(x, np.float32)).to(torch.bfloat16).view(
        torch.int16).numpy().view(np.uint16)


def near(q, others, most):
    """Unit rows around q, nearer and farther."""
    x = bf16_f64(q)[None] + np.linspace(0.02, most, len(others))[:, None] * bf16_f64(others)
    return bits(x / np.linalg.norm(x, axis=1, keepdims=True))


def dev(x):
    return to_dev(x).view(torch.bfloat16)


def best(Q, C, k):
    """Scores and ids in order; scores that are equal in 64 bits by lower id."""
    full = bf16_f64(Q) @ bf16_f64(C).T
    order = np.lexsort((np.broadcast_to(np.arange(len(C)), full.shape), -full))[:, :k]
    return full, np.take_along_axis(full, order, 1), order


def same(s, i, full, want, rows=slice(None)):
    s, i = s.cpu().numpy(), i.cpu().numpy().astype(np.int64)
    assert np.abs(s - want[rows]).max() < 1e-3
    assert np.abs(np.take_along_axis(full[rows], i, 1) - want[rows]).max() < 1e-3
    assert all(len(set(r)) == i.shape[1] for r in i.tolist())


# 40,000 rows are 157 tiles of 256, each of two halves that are lists of their own.
@pytest.mark.parametrize("at", [2 * 256 + 8, 2 * 256 + 100, 3 * 256 - 30, 40000 - 60])
@pytest.mark.parametrize("k", [17, 32, 40, 100])
@pytest.mark.parametrize("nq", [6, 65, 130, 300])
def test_identical_neighbours(nq, k, at):
    """60 bit-identical best rows inside one list, over two, over two tiles and at
    the end: every score at the floor is a tie, and the lowest ids win."""
    C = synth.unit_rows(40000, 128, 3)
    Q = synth.unit_rows(nq, 128, 4)
    C[at:at + 60] = Q[nq // 2]
    s, i = hs.hs_retrieve_topk(dev(Q), dev(C), k)
    hs.hs_get_device_error()
    rows = [0, nq // 2, nq - 1]
    full, want, order = best(Q[rows], C, k)
    same(s[rows], i[rows], full, want)
    first = min(k, 60)
    assert i[nq // 2, :first].tolist() == list(range(at, at + first))


@pytest.mark.parametrize("k", [17, 24, 32, 33, 64])
@pytest.mark.parametrize("nq", [20, 200, 700])
def test_every_query_crowded(nq, k):
    """Every query's best rows side by side, queries by the hundred in one list."""
    C = synth.unit_rows(20000, 64, k)
    Q = synth.unit_rows(nq, 64, 6)
    Q[nq // 2:] = Q[0]                               # half of them meet in the same lists
    for j in range(nq // 2):
        p = 19900 // (nq // 2) * j
        C[p:p + 25] = near(Q[j], C[:25], 0.4)
    s, i = hs.hs_retrieve_topk(dev(Q), dev(C), k)
    hs.hs_get_device_error()
    full, want, _ = best(Q, C, k)
    same(s, i, full, want)


@pytest.mark.parametrize("crowd", [25, 50])
@pytest.mark.parametrize("k", [20, 40])
def test_device_count_fanout_and_a_bad_entry(k, crowd):
    """A count below max_queries, several rows per cut query, and one entry of the
    map out of range, which is reported while all other rows are right."""
    rng = np.random.default_rng(k)
    C = synth.unit_rows(30000, 128, k)
    Q = synth.unit_rows(400, 128, 6)
    live = 260
    for j in range(0, live, 5):
        p = 500 * (j // 5) + 90
        C[p:p + crowd] = near(Q[j], C[:crowd], 0.4) if j % 2 else Q[j]
    inv = rng.integers(0, live, size=900).astype(np.int32)
    inv[77] = live                                   # a query past the count
    dq, dc = dev(Q), dev(C)
    s = torch.full((900, k), 7.0, device="cuda")
    i = torch.full((900, k), 7, dtype=torch.int32, device="cuda")
    hs.hs_retrieve_topk_fanout(dq, to_dev(np.array([live], np.int32)), to_dev(inv), dc, k,
                               out=(s, i))
    with pytest.raises(hs.HsError) as e:
        hs.hs_get_device_error()
    assert e.value.status == hs.HS_ERR_INVALID_ARG
    assert (s[77] == 7.0).all() and (i[77] == 7).all()
    ok = np.arange(900) != 77
    full, want, _ = best(Q[:live], C, k)
    same(s[torch.from_numpy(ok)], i[torch.from_numpy(ok)], full[inv[ok]], want[inv[ok]])


@pytest.mark.parametrize("nq,N,k", [(3, 20000, 200), (20, 20000, 33), (140, 9000, 300)])
def test_all_rows_equal(nq, N, k):
    """Every row ties at the floor: lists cut everywhere and cut again."""
    C = np.tile(synth.unit_rows(1, 64, 1), (N, 1))
    s, i = hs.hs_retrieve_topk(dev(np.tile(synth.unit_rows(1, 64, 2), (nq, 1))), dev(C), k)
    hs.hs_get_device_error()
    assert (i.cpu().numpy() == np.arange(k)).all() and (s == s[0, 0]).all()


@pytest.mark.parametrize("k", [20, 50])
def test_zero_rows_of_both_signs(k):
    """Queries and rows of all-zero and all-negative-zero scores tie with one another."""
    C = np.zeros((9000, 64), np.uint16)
    C[::2] = 0x8000                                  # -0.0
    Q = np.full((5, 64), 0x8000, np.uint16)
    Q[1] = 0
    Q[2:] = synth.unit_rows(3, 64, 1)
    s, i = hs.hs_retrieve_topk(dev(Q), dev(C), k)
    hs.hs_get_device_error()
    assert (s == 0).all() and (i.cpu().numpy() == np.arange(k)).all()


def test_scores_do_not_depend_on_the_batch():
    """A floor of one pass is compared with scores of another: 1 to 300 queries, by
    every variant of the kernel, get the same bits."""
    C, Q = dev(synth.unit_rows(30000, 776, 1)), dev(synth.unit_rows(300, 776, 2))
    for k in (10, 24, 50, 300):
        want = hs.hs_retrieve_topk(Q, C, k)
        for n in (1, 17, 64, 65, 129):
            got = hs.hs_retrieve_topk(Q[:n].contiguous(), C, k)
            assert torch.equal(got[0], want[0][:n]) and torch.equal(got[1], want[1][:n])
    hs.hs_get_device_error()


@pytest.mark.parametrize("k", [24, 50])
def test_wait_runs_out_with_cut_lists(k):
    Q, C = synth.unit_rows(200, 128, 3), synth.unit_rows(30000, 128, 4)
    C[1000:1030] = Q[7]
    Q, C = dev(Q), dev(C)
    want = hs.hs_retrieve_topk(Q, C, k)
    try:
        hs.hs_debug_retrieve_wait(1_000_000, 1)
        hs.hs_retrieve_topk(Q, C, k)
        with pytest.raises(hs.HsError) as e:
            hs.hs_get_device_error()
        assert e.value.status == hs.HS_ERR_TIMEOUT
    finally:
        hs.hs_debug_retrieve_wait()
    got = hs.hs_retrieve_topk(Q, C, k)
    hs.hs_get_device_error()
    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])


def test_cut_lists_cost_their_own_rows():
    """300 queries whose 20 best rows are neighbours, k = 17, against the same batch
    on a corpus in random order: 1.4 times the time (2.5 times with a second pass of
    32 slots over the whole corpus for the cut queries; 1.9 is halfway)."""
    C, Q = synth.unit_rows(131072, 384, 1), synth.unit_rows(300, 384, 2)
    crowded = C.copy()
    for j in range(300):
        p = 436 * j + 145
        crowded[p:p + 20] = near(Q[j], C[:20], 0.5)
    dq, k = dev(Q), 17
    us = []
    for c in (dev(C), dev(crowded)):
        ws = torch.empty(hs.hs_retrieve_topk_workspace(300, 131072, 384, k), dtype=torch.uint8,
                         device="cuda")
        out = (torch.empty((300, k), device="cuda"),
               torch.empty((300, k), dtype=torch.int32, device="cuda"))
        us.append(graph_us(lambda: hs.hs_retrieve_topk(dq, c, k, workspace=ws, out=out)))
    hs.hs_get_device_error()
    assert us[1] < 1.9 * us[0], us


def test_many_results_for_few_queries():
    """The merge of more than 128 results takes a round per result, by the number of
    lists: wide rows (1024), whose ring allows tiles of 128 only, do not get more of
    them than rows of 768 (1.24 times the time with twice as many; 1.02 without)."""
    us = []
    for d in (768, 1024):
        q, c = dev(synth.unit_rows(3, d, 1)), dev(synth.unit_rows(32768, d, 2))
        ws = torch.empty(hs.hs_retrieve_topk_workspace(3, 32768, d, 500), dtype=torch.uint8,
                         device="cuda")
        out = (torch.empty((3, 500), device="cuda"),
               torch.empty((3, 500), dtype=torch.int32, device="cuda"))
        us.append(graph_us(lambda: hs.hs_retrieve_topk(q, c, 500, workspace=ws, out=out)))
    hs.hs_get_device_error()
    assert us[1] < 1.12 * us[0], us
