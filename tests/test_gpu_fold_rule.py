"""Which kernel a matrix of the fp32 product takes (table lookups or tensor cores), at both
sides of each line: against 64 bits from the same codes and centres, and the same bits alone,
in a call with matrices of the other side, and (lookups) in fewer rows.

Tolerance, per row, of max |Y|: 1e-5, that of test_gpu_fold."""

import pytest
import torch

from tests.test_gpu_fold import TOL, kd  # noqa: F401  (the module's fixture)
from tests.test_gpu_fold_tc import _case, _y64

pytestmark = pytest.mark.gpu

# n, m, batch, whether the lookup kernel takes it
LINES = [(1024, 3073, 2, True), (1000, 3072, 2, True), (1000, 3073, 2, False),
         (4096, 512, 3, True), (4096, 513, 4, False), (4095, 60, 3, False),
         (4096, 341, 5, True), (4096, 129, 16, False), (4096, 128, 15, True), (4096, 16, 17, False),
         (11008, 1, 16, True)]


@pytest.mark.parametrize("n,m,batch,lookup", LINES)
@pytest.mark.parametrize("kmeans", [0, 1])
def test_both_sides(kd, n, m, batch, lookup, kmeans):  # noqa: F811
    dec, x, xp = _case(kd, n, m, batch, kmeans)
    y = kd.matmul_2bit(dec, x, xp)
    ref = _y64(dec, x, xp)
    err = (y.double() - ref).abs().amax(1) / ref.abs().amax(1).clamp(min=ref.abs().mean())
    assert (err <= TOL).all(), err.max().item()
    one = torch.cat([kd.matmul_2bit(dec, x[r:r + 1], xp[r:r + 1]) for r in range(batch)])
    assert torch.equal(y, one) == lookup  # one row is always looked up: the bits tell the kernels apart
    d2, x2, xp2 = _case(kd, 300, 5000, batch, kmeans)
    d3, x3, xp3 = _case(kd, 4096, 100, batch, kmeans)
    ys = kd.matmul_2bit_batch([d2, dec, d3], [x2, x, x3], [xp2, xp, xp3])
    assert torch.equal(ys[1], y)
    assert torch.equal(ys[0], kd.matmul_2bit(d2, x2, xp2)) and torch.equal(ys[2], kd.matmul_2bit(d3, x3, xp3))


def test_lookup_rows_at_odd_strides(kd):  # noqa: F811
    """Five rows (the last pair half empty) at an odd offset and stride: the bits of the
    contiguous call, nothing written beside them."""
    dec, x, xp = _case(kd, 4096, 70, 5)
    ref = kd.matmul_2bit(dec, x, xp)
    big = torch.zeros((2, 5, 4139), device="cuda")
    xs, ps = big[0][:, 1:4097], big[1][:, 1:4097]
    xs.copy_(x)
    ps.copy_(xp)
    ys = torch.full((6, 75), float("nan"), device="cuda")
    kd.matmul_2bit(dec, xs, ps, out=ys[:5, :70])
    assert torch.equal(ys[:5, :70], ref)
    assert torch.isnan(ys[5]).all() and torch.isnan(ys[:, 70:]).all()
