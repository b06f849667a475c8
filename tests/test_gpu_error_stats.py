"""The FP64 error reduction over its index arithmetic and launch sizes: group
divisors, ragged and unaligned lengths, runs of one and of many CTAs, against
numpy FP64 (1e-12 relative for the sums, the exact maximum without weights)."""
import math

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def expected(a, b, w, group, stride):
    a, b = a.astype(np.float64), b.astype(np.float64)
    k = 1.0 if w is None else w.astype(np.float64)[(np.arange(len(a)) // group) * stride]
    d, e = k * (a - b), k * b
    return np.array([np.sum(d * d), np.sum(e * e), np.max(np.abs(d))])


@pytest.mark.parametrize("group,stride", [(1, 1), (2, 1), (3, 3), (5, 2), (7, 1), (64, 1), (1000, 1), (65537, 1)])
@pytest.mark.parametrize("n,offset", [(1, 0), (2, 0), (777, 0), (311297, 0), (1245185, 1), (2500001, 0)])
def test_group_divisors_and_sizes(fab, group, stride, n, offset):
    r = np.random.default_rng([group, n])
    a = r.standard_normal(n + offset).astype(np.float32)
    b = (a + 0.1 * r.standard_normal(n + offset)).astype(np.float32)
    w = r.uniform(0.1, 1.0, ((n - 1) // group) * stride + 1).astype(np.float32)
    da, db, dw = (torch.from_numpy(x).cuda() for x in (a, b, w))
    got = fab.error_stats(da[offset:], db[offset:], weights=dw, group=group, weight_stride=stride).cpu().numpy()
    want = expected(a[offset:], b[offset:], w, group, stride)
    assert np.all(np.abs(got - want) <= 1e-12 * want)
    got = fab.error_stats(da[offset:], db[offset:]).cpu().numpy()
    want = expected(a[offset:], b[offset:], None, 1, 1)
    assert np.all(np.abs(got[:2] - want[:2]) <= 1e-12 * want[:2]) and got[2] == want[2]


def test_calls_at_once_leave_nothing_behind(fab):
    """Three sizes on three streams at once may spoil each other (they share
    the partial sums), but a call alone afterwards, on other values, is right:
    nothing that one call counts or leaves is read by another."""
    r = np.random.default_rng(11)

    def arrays(n):
        a = r.standard_normal(n).astype(np.float32)
        b = (a + 0.1 * r.standard_normal(n)).astype(np.float32)
        return torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda(), expected(a, b, None, 1, 1)

    sizes = (1000, 311297, 1 << 22)
    at_once = [arrays(n) for n in sizes]
    alone = [arrays(n) for n in sizes]
    streams = [torch.cuda.Stream() for _ in sizes]
    out = torch.empty(3, dtype=torch.float64, device="cuda")
    for _ in range(20):
        torch.cuda.synchronize()
        for s, (a, b, _) in list(zip(streams, at_once)) * 10:
            fab.error_stats(a, b, out=out, stream=s)
        torch.cuda.synchronize()
        for a, b, want in alone:
            got = fab.error_stats(a, b, out=torch.full((3,), float("nan"), dtype=torch.float64, device="cuda"))
            assert np.all(np.abs(got.cpu().numpy() - want) <= 1e-12 * want)


@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("n", [1000, 311297])
def test_products_below_the_fp32_range(fab, n, offset):
    """Weights whose products with the differences, or with b, vanish in FP32
    still count, on the packed and on the scalar path; so do zero weights and
    equal values for nothing."""
    r = np.random.default_rng(n)
    b = (2.0 ** -58 * r.uniform(1.0, 2.0, n + offset)).astype(np.float32)
    a = (b * r.uniform(1.0, 2.0, n + offset)).astype(np.float32)
    w = (2.0 ** -100 * r.uniform(1.0, 2.0, n)).astype(np.float32)
    w[::3] = 0.0
    a[::4] = b[::4]
    da, db, dw = (torch.from_numpy(x).cuda() for x in (a, b, w))
    got = fab.error_stats(da[offset:], db[offset:], weights=dw).cpu().numpy()
    want = expected(a[offset:], b[offset:], w, 1, 1)
    assert np.all(want > 0.0) and np.all(np.abs(got - want) <= 1e-12 * want)


def test_sums_round_only_in_fp64(fab):
    """FP32 values with all 24 bits in use and a = -b, so that every term is
    exact in FP64, one pair to a thread: what is left are the roundings of a
    tree of FP64 additions, at most 22 in sequence, each at most 2^-53 of the
    sum and to either side.  Rounded anywhere to the 48 bits of an FP32 pair
    the sums come out low (odd squares are 1 modulo 4, so their ties all fall
    the same way).  A call's error is then below sqrt(22 / 3) 2^-53 = 3.0e-16
    rms, the mean over 40 calls within three standard deviations of zero below
    1.43e-16."""
    n, calls = 50001, 40
    err = np.zeros(2)
    for k in range(calls):
        b = np.random.default_rng([5, k]).random(n).astype(np.float32)
        got = fab.error_stats(torch.from_numpy(-b).cuda(), torch.from_numpy(b).cuda()).cpu().numpy()
        want = math.fsum(b.astype(np.float64) ** 2)
        for j, scale in enumerate((0.25, 1.0)):
            err[j] += math.fsum([scale * float(got[j]), -want]) / want / calls
    assert np.all(np.abs(err) < 1.43e-16), err
