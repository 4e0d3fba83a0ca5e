"""Fingerprints (Section 3.3, Eq. 2) and the exact merge (Section 3.3 (I)) at
the edges of the 32-token chunks and 16-byte pieces: every word offset of a
row's start, lengths around them, both ends of the token array, tokens above
and below 65536."""
import numpy as np
import pytest
import torch

import oracle
import paper_2607_22578_gb300 as hs
from hs_testutil import graph_us, to_dev

pytestmark = pytest.mark.gpu


def rows_at(offset, n, stride, rng, big):
    """n rows whose first word lies `offset` words past a 256-byte boundary,
    in an array with nothing after its last word."""
    flat = rng.integers(0, 1 << 31 if big else 65536, size=offset + n * stride).astype(np.int32)
    dev = to_dev(flat)
    return flat[offset:].reshape(n, stride), dev[offset:].view(n, stride)


@pytest.mark.parametrize("big", [False, True])
@pytest.mark.parametrize("stride", [1, 3, 4, 7, 8, 31, 32, 33, 36, 63, 64, 65, 96, 333])
def test_fingerprint_at_every_offset(stride, big):
    rng = np.random.default_rng(stride + big)
    for offset in range(9):
        tokens, dev = rows_at(offset, 77, stride, rng, big)
        lens = rng.integers(0, stride + 1, size=77).astype(np.int32)
        lens[[0, 76]] = stride                       # the array's first and last words
        for L in (None, lens):
            for seed in (hs.HS_FNV64_OFFSET_BASIS, 0x0123456789ABCDEF):
                fp = hs.hs_fingerprint(dev, None if L is None else to_dev(L), seed)
                hs.hs_get_device_error()
                want = oracle.fingerprint(tokens, L, seed=seed)
                assert (fp.cpu().numpy().view(np.uint64) == want).all(), (offset, L is None)


@pytest.mark.parametrize("big", [False, True])
@pytest.mark.parametrize("stride", [1, 8, 33, 255, 256, 257, 513, 1280])
def test_fingerprint_on_both_sides_of_the_row_count(stride, big):
    """Few rows are hashed by a warp each (1024 octets at a time), many by a
    lane each."""
    rng = np.random.default_rng(stride + big)
    for offset, n in ((0, 1), (0, 33), (1, 33), (0, 13000), (3, 13000)):
        tokens, dev = rows_at(offset, n, stride, rng, big)
        lens = rng.integers(0, stride + 1, size=n).astype(np.int32)
        lens[[0, n - 1]] = stride
        for L in (None, lens):
            fp = hs.hs_fingerprint(dev, None if L is None else to_dev(L), 0xFFFFFFFFFFFFFFFF)
            hs.hs_get_device_error()
            want = oracle.fingerprint(tokens, L, seed=0xFFFFFFFFFFFFFFFF)
            assert (fp.cpu().numpy().view(np.uint64) == want).all(), (offset, n)


@pytest.mark.parametrize("stride", [2, 8, 9, 12, 16, 17, 20, 24, 25, 28, 31])
@pytest.mark.parametrize("offset", [0, 1])
def test_fingerprint_of_rows_shorter_than_a_chunk(offset, stride):
    """A thread per row, with room for 8, 16, 24 or 32 tokens; few rows of more than
    16 by a warp each."""
    rng = np.random.default_rng(stride)
    for n in (3, 700, 5003):
        tokens, dev = rows_at(offset, n, stride, rng, bool(n % 2))
        lens = rng.integers(0, stride + 1, size=n).astype(np.int32)
        lens[[0, n - 1]] = stride
        for L in (None, lens):
            want = oracle.fingerprint(tokens, L)
            fp = hs.hs_fingerprint(dev, None if L is None else to_dev(L))
            hs.hs_get_device_error()
            assert (fp.cpu().numpy().view(np.uint64) == want).all(), (n, L is None)
        bad = lens.copy()
        bad[1] = stride + 1
        fp = hs.hs_fingerprint(dev, to_dev(bad))
        with pytest.raises(hs.HsError):
            hs.hs_get_device_error()
        want[1] = 0
        assert (fp.cpu().numpy().view(np.uint64) == want).all()


@pytest.mark.parametrize("n,stride", [(7000, 644), (16384, 512), (16384, 200), (80001, 256),
                                      (80001, 36), (16383, 508), (80000, 252)])
def test_fingerprint_in_two_passes(n, stride):
    """Aligned rows of which many have full chunks: chunks first, then the rests;
    and beside each rule's line, in one pass."""
    rng = np.random.default_rng(stride)
    tokens, dev = rows_at(0, n, stride, rng, False)
    lens = rng.integers(0, stride + 1, size=n).astype(np.int32)
    lens[:4] = [0, 32, stride, 31]
    for L in (None, lens):
        fp = hs.hs_fingerprint(dev, None if L is None else to_dev(L), 7)
        hs.hs_get_device_error()
        assert (fp.cpu().numpy().view(np.uint64) == oracle.fingerprint(tokens, L, seed=7)).all()
    bad = lens.copy()
    bad[[1, n - 1]] = [-5, stride + 32]
    fp = hs.hs_fingerprint(dev, to_dev(bad), 7)
    with pytest.raises(hs.HsError) as e:
        hs.hs_get_device_error()
    assert e.value.status == hs.HS_ERR_INVALID_ARG
    want = oracle.fingerprint(tokens, lens, seed=7)
    want[[1, n - 1]] = 0
    assert (fp.cpu().numpy().view(np.uint64) == want).all()


def _ragged_us(n, stride, low):
    t = torch.zeros((n, stride), dtype=torch.int32, device="cuda")
    lens = torch.randint(low, stride + 1, (n,), dtype=torch.int32, device="cuda")
    fp = torch.empty(n, dtype=torch.int64, device="cuda")
    return graph_us(lambda: hs.hs_fingerprint(t, lens, fp_out=fp))


def test_short_rows_cost_no_chunk():
    """A million rows of up to 8 tokens take less than the half of as many of 24 to 28
    (0.28; 0.56 where each took a lane's chunk)."""
    assert _ragged_us(1000000, 8, 1) < 0.43 * _ragged_us(1000000, 28, 24)


def test_long_ragged_rows_cost_no_masks():
    """40,000 rows of up to 2048 tokens against as many of exactly 1024: 2.05 times the
    time (2.5 times where every chunk is masked; the longest chain is twice as long)."""
    t = torch.zeros((40000, 1024), dtype=torch.int32, device="cuda")
    fp = torch.empty(40000, dtype=torch.int64, device="cuda")
    whole = graph_us(lambda: hs.hs_fingerprint(t, fp_out=fp))
    assert _ragged_us(40000, 2048, 1) < 2.25 * whole, whole


def test_fingerprint_mixes_small_and_large_tokens_and_bad_lengths():
    rng = np.random.default_rng(9)
    tokens, dev = rows_at(2, 5000, 75, rng, False)
    tokens = tokens.copy()
    tokens[rng.random(tokens.shape) < 0.01] = -1     # some chunks take the octet-wise rounds
    dev.copy_(to_dev(tokens))
    lens = rng.integers(0, 76, size=5000).astype(np.int32)
    want = oracle.fingerprint(tokens, lens)
    bad = lens.copy()
    bad[[0, 31, 4999]] = [-1, 76, 1 << 30]
    fp = hs.hs_fingerprint(dev, to_dev(bad))
    with pytest.raises(hs.HsError) as e:
        hs.hs_get_device_error()
    assert e.value.status == hs.HS_ERR_INVALID_ARG
    want[[0, 31, 4999]] = 0
    assert (fp.cpu().numpy().view(np.uint64) == want).all()


@pytest.mark.parametrize("stride", [1, 5, 33, 127, 130])
def test_merge_of_rows_on_any_word(stride):
    rng = np.random.default_rng(stride)
    n = 4097 + stride
    for offset in (0, 1, 3):
        tokens, dev = rows_at(offset, n, stride, rng, True)
        tokens = tokens.copy()
        src = rng.integers(0, n, size=n)
        copy = rng.random(n) < 0.5
        tokens[copy] = tokens[src[copy]]
        near = rng.integers(0, n, size=n // 8)       # rows that differ in one word only
        tokens[near] = tokens[0]
        tokens[near, rng.integers(0, stride, size=len(near))] ^= 1 << 20
        dev.copy_(to_dev(tokens))
        lens = np.where(rng.random(n) < 0.5, stride, rng.integers(0, stride + 1, size=n))
        lens = lens.astype(np.int32)
        for L in (None, lens):
            d = None if L is None else to_dev(L)
            ou, oi = oracle.unique_inverse(tokens, L)
            fp, nu, u, i = hs.hs_merge_rows(dev, d)
            nu2, u2, i2 = hs.hs_unique_inverse(fp, dev, d)
            hs.hs_get_device_error()
            assert (fp.cpu().numpy().view(np.uint64) == oracle.fingerprint(tokens, L)).all()
            for count, uniq, inv in ((nu, u, i), (nu2, u2, i2)):
                assert int(count.item()) == len(ou)
                assert (uniq.cpu().numpy()[:len(ou)] == ou).all()
                assert (uniq.cpu().numpy()[len(ou):] == 0).all()
                assert (inv.cpu().numpy() == oi).all()


def test_few_unaligned_rows_have_a_warp_each():
    """8192 unaligned rows of 2048 tokens against as many aligned ones, which have a
    lane each: 1.15 times (2.3 times with a lane each)."""
    us = []
    for offset in (0, 1):
        t = torch.zeros(8192 * 2048 + offset, dtype=torch.int32, device="cuda")
        rows = t[offset:].view(8192, 2048)
        fp = torch.empty(8192, dtype=torch.int64, device="cuda")
        us.append(graph_us(lambda: hs.hs_fingerprint(rows, fp_out=fp)))
    assert us[1] < 1.7 * us[0], us
