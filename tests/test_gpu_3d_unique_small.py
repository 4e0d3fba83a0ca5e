"""The one-launch unique (Section 3.3 (I)) at the edges of its cluster: row
counts around a CTA's share, the CTA counts and the two block sizes, collisions
in every CTA's share, invalid lengths, and its use of a workspace whose
contents are anything."""
import numpy as np
import pytest
import torch

import oracle
import paper_2607_22578_gb300 as hs
from hs_testutil import graph_us, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("stride", [3, 8, 100])
@pytest.mark.parametrize("n", [1, 8, 63, 64, 65, 128, 129, 257, 512, 513, 2047, 2048, 2049, 4095, 4096])
def test_row_counts(n, stride):
    rng = np.random.default_rng(n + stride)
    tokens = rng.integers(0, 1 << 31, size=(n, stride)).astype(np.int32)
    src = rng.integers(0, n, size=n)
    copy = rng.random(n) < 0.6
    tokens[copy] = tokens[src[copy]]
    lens = np.where(rng.random(n) < 0.5, stride, rng.integers(0, stride + 1, size=n)).astype(np.int32)
    t = to_dev(tokens)
    ws = torch.full((hs.hs_unique_inverse_workspace(n),), 0x5A, dtype=torch.uint8, device="cuda")
    for L in (None, lens):
        d = None if L is None else to_dev(L)
        ou, oi = oracle.unique_inverse(tokens, L)
        fp = hs.hs_fingerprint(t, d)
        few = fp % 5                                 # equal rows alike, most others too
        for key in (fp, few, torch.zeros_like(fp)):
            nu, u, inv = hs.hs_unique_inverse(key, t, d, workspace=ws)
            hs.hs_get_device_error()
            assert int(nu.item()) == len(ou)
            assert (u.cpu().numpy()[:len(ou)] == ou).all() and (u.cpu().numpy()[len(ou):] == 0).all()
            assert (inv.cpu().numpy() == oi).all()


@pytest.mark.parametrize("n", [4097, 8191, 8193, 70001])
def test_workspace_cleared(n):
    """Above one cluster: counters, scan states and the table's last slot
    (fingerprint of all ones) come out of the clearing launch."""
    rng = np.random.default_rng(n)
    tokens = rng.integers(0, 50, size=(n, 4)).astype(np.int32)
    tokens[n // 2:] = tokens[rng.integers(0, n // 2, size=n - n // 2)]
    t = to_dev(tokens)
    ou, oi = oracle.unique_inverse(tokens, None)
    fp = hs.hs_fingerprint(t)
    ones = torch.where(t[:, 0] < 1, torch.full_like(fp, -1), fp)
    for fill in (0x00, 0x5A, 0xFF):
        ws = torch.full((hs.hs_merge_rows_workspace(n),), fill, dtype=torch.uint8, device="cuda")
        calls = [lambda k=k: hs.hs_unique_inverse(k, t, workspace=ws) for k in (fp, ones)]
        for call in calls + [lambda: hs.hs_merge_rows(t, workspace=ws)[-3:]]:
            nu, u, inv = call()
            hs.hs_get_device_error()
            assert int(nu.item()) == len(ou)
            assert (u.cpu().numpy()[:len(ou)] == ou).all() and (inv.cpu().numpy() == oi).all()


def test_many_unaligned_rows_cost_little_more():
    """A million rows of 31 words, hardly one a copy, against as many of 32: 1.09 times
    the time, which is lookups mostly (1.20 with twice the words in flight per lane, and
    fewer warps for it)."""
    us = []
    for stride in (31, 32):
        g = torch.Generator(device="cuda").manual_seed(1)
        rows = torch.randint(0, 1 << 30, (1000000, stride), dtype=torch.int32, device="cuda",
                             generator=g)
        fp = hs.hs_fingerprint(rows)
        ws = torch.empty(hs.hs_unique_inverse_workspace(len(rows)), dtype=torch.uint8,
                         device="cuda")
        out = tuple(torch.empty(k, dtype=torch.int32, device="cuda") for k in (1, len(rows),
                                                                               len(rows)))
        us.append(graph_us(lambda: hs.hs_unique_inverse(fp, rows, workspace=ws, out=out)))
    assert us[0] < 1.15 * us[1], us
