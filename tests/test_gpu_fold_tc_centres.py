"""The products from the 2-bit planes with centres that are far from symmetric about 0, in one
row (table lookups) and in more (tensor cores), against 64 bits from the same codes and centres.

Tolerance, per output: 1e-6 of the sum of its terms' magnitudes.  Each sum of the inputs of one
code is exact to fp32 and takes at most 12 fp32 roundings (2^-24 each) of values no larger than
that sum of magnitudes on its way into the result; the lookup kernel's sums of up to 64 terms
per lane have 96 roundings of partial sums, far below it at these sizes."""

import pytest
import torch

from tests.test_gpu_fold import kd  # noqa: F401  (the module's fixture)
from tests.test_gpu_fold_tc import _case, _plane, _y64

pytestmark = pytest.mark.gpu


def _recode(codes, j, old, new):
    """Channel j's codes `old` become `new`."""
    w = codes[j].long() & 0xFFFFFFFF
    q = w.unsqueeze(1) >> (2 * torch.arange(16, device=codes.device)) & 3
    q[q == old] = new
    w = (q << (2 * torch.arange(16, device=codes.device))).sum(1)
    codes[j] = torch.where(w > 0x7FFFFFFF, w - (1 << 32), w).int()


@pytest.mark.parametrize("batch", [1, 2, 16, 17])
@pytest.mark.parametrize("n", [300, 4096])
def test_centres_far_from_symmetric(kd, n, batch):  # noqa: F811
    dec, x, xp = _case(kd, n, 140, batch)
    cu, cv = dec.centres_u, dec.centres_v
    cu[3] = torch.tensor([-1.0, -0.3, 0.3, 1e8])          # the largest centre unused
    _recode(dec.codes_u, 3, 3, 2)
    cu[4] = torch.tensor([-1e8, -0.3, 0.2, 1.0])          # the lowest unused
    _recode(dec.codes_u, 4, 0, 1)
    cu[5] = torch.tensor([-1.0, -0.3, 0.3, 2.0 ** 100])   # just below the plain sums' line, unused
    _recode(dec.codes_u, 5, 3, 2)
    cv[6] = torch.tensor([-1.0, -1e-6, 1e-3, 1e3])        # both pairs unequal, all used
    cv[7] = torch.tensor([1.0, 2.0, 3.0, 4.0])            # all of one sign
    cv[8] = torch.tensor([-1e8, -1e8, 1.0, 1.0])          # an inner centre unused
    _recode(dec.codes_v, 8, 1, 2)
    _recode(dec.codes_v, 8, 0, 3)
    cu[139] = torch.tensor([-1.0, -0.6, 1.0, 1.7])        # on both sides of the line
    cv[139] = torch.tensor([-1.0, -0.59, 1.0, 1.6])
    y = kd.matmul_2bit(dec, x, xp)
    ref = _y64(dec, x, xp)
    size = x.double().abs() @ _plane(dec.codes_u, cu, n).abs().t() + xp.double().abs() @ _plane(dec.codes_v, cv, n).abs().t()
    assert torch.isfinite(y).all()
    err = ((y.double() - ref).abs() / size).amax(0)
    assert (err <= 1e-6).all(), (err.argmax().item(), err.max().item())


@pytest.mark.parametrize("batch", [2, 16])
def test_a_huge_sum_beside_a_huge_unused_centre(kd, batch):  # noqa: F811
    """2^100 unused beside sums of 2^40: finite results, the same as in one row."""
    dec, x, xp = _case(kd, 300, 140, batch)
    x *= 2.0 ** 40
    dec.centres_u[9] = torch.tensor([-1.0, -0.3, 0.3, 2.0 ** 100])
    _recode(dec.codes_u, 9, 3, 2)
    y = kd.matmul_2bit(dec, x, xp)
    one = torch.cat([kd.matmul_2bit(dec, x[r:r + 1], xp[r:r + 1]) for r in range(batch)])
    assert torch.isfinite(y).all()
    err = (y.double() - one.double()).abs() / (x.double().abs() @ _plane(dec.codes_u, dec.centres_u, 300).abs().t())
    assert (err <= 2e-6).all(), err.max().item()
