"""hs_merge_queries groups rows by a key of its own and hashes them beside the
merge (Section 3.3, Eq. 2 and (I)): widths around the lane groups that share a
row, rows that differ in a single place, every way to pass fingerprints."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
import paper_2607_22578_gb300 as hs
from hs_testutil import to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [8, 16, 24, 64, 248, 256, 264, 768, 776, 2056])
@pytest.mark.parametrize("n", [1, 2, 33, 255, 256])
def test_widths_and_near_rows(n, d):
    rng = np.random.default_rng(n * 7 + d)
    q = np.tile(rng.integers(0, 1 << 16, size=d, dtype=np.uint16), (n, 1))
    for i in range(0, n, 2):                    # half the rows differ in one place, some twice
        q[i, (i * 5) % d] ^= 1 + i // (2 * d)
    q[n // 2] = q[0]
    fp, nu, u, inv, uq = hs.hs_merge_queries(to_dev(q), 12345)
    hs.hs_get_device_error()
    ou, oi = oracle.unique_inverse(np.ascontiguousarray(q).view(np.int32))
    k = int(nu.item())
    assert k == len(ou) and (u.cpu().numpy()[:k] == ou).all() and (u.cpu().numpy()[k:] == 0).all()
    assert (inv.cpu().numpy() == oi).all()
    assert (uq[:k].cpu().view(torch.int16).numpy().view(np.uint16) == q[ou]).all()
    want = oracle.fingerprint(np.ascontiguousarray(q).view(np.int32), None, seed=12345)
    assert (fp.cpu().numpy().view(np.uint64) == want).all()


@pytest.mark.parametrize("given", [False, True])
@pytest.mark.parametrize("asked", [False, True])
def test_fingerprints_given_and_asked_for(given, asked):
    rng = np.random.default_rng(3)
    q = rng.integers(0, 3, size=(97, 16), dtype=np.uint16)
    q[:, 1:] = 0
    t = to_dev(q)
    fp_in = torch.arange(97, dtype=torch.int64, device="cuda") * 0 + 7     # all alike
    out = [torch.zeros(97, dtype=torch.int64, device="cuda"),
           *(torch.empty(m, dtype=torch.int32, device="cuda") for m in (1, 97, 97)),
           torch.empty_like(t)]
    p = [None if x is None else ctypes.c_void_p(x.data_ptr()) for x in
         (fp_in if given else None, out[0] if asked else None, *out[1:])]
    st = hs.load().hs_merge_queries(t.data_ptr(), 97, 16, 99, *p,
                                    torch.cuda.current_stream().cuda_stream)
    assert st == hs.HS_OK
    hs.hs_get_device_error()
    ou, oi = oracle.unique_inverse(q.view(np.int32))
    assert int(out[1].item()) == len(ou) and (out[3].cpu().numpy() == oi).all()
    want = np.full(97, 7, np.uint64) if given else oracle.fingerprint(q.view(np.int32), None, seed=99)
    got = out[0].cpu().numpy().view(np.uint64)
    assert (got == (want if asked else 0)).all()
