"""The fp32 product from the 2-bit planes on the tensor cores (two batch rows and more) over
inputs whose magnitudes differ widely, against 64 bits from the same codes and centres.

Tolerance, per row, of max |Y|: 1e-6, as in test_gpu_fold_tc.  The sums of the inputs' digits
are exact to 2^-32 of the row's largest input each; after them come at most 12 fp32 roundings
of values up to a few max |Y| (per plane and part three additions of the digits, two products
and their sum; then the parts)."""

import pytest
import torch

from tests.test_gpu_fold import kd  # noqa: F401  (the module's fixture)
from tests.test_gpu_fold_tc import _case, _plane, _y64

pytestmark = pytest.mark.gpu

TOL = 1e-6


def _check(y, ref):
    err = (y.double() - ref).abs().amax(1) / ref.abs().amax(1)
    assert (err <= TOL).all(), err.max().item()


@pytest.mark.parametrize("n,batch", [(256, 2), (768, 33), (4096, 16), (11008, 17)])
@pytest.mark.parametrize("e", [10, 18, 26])
def test_one_input_leads_the_row(kd, n, batch, e):  # noqa: F811
    """One input 2^e times the others, at the first, the last or another place of the row."""
    dec, x, xp = _case(kd, n, 130, batch)
    for r in range(batch):
        x[r, (0, n - 1, (37 * r) % n)[r % 3]] = 1.2345678 * 2.0 ** e
    _check(kd.matmul_2bit(dec, x, xp), _y64(dec, x, xp))


@pytest.mark.parametrize("n,batch", [(256, 33), (4096, 16), (11008, 5)])
def test_log_normal_inputs(kd, n, batch):  # noqa: F811
    dec, x, xp = _case(kd, n, 130, batch, kmeans=1)
    g = torch.Generator(device="cuda").manual_seed(n)
    x *= torch.exp(2 * torch.randn(x.shape, generator=g, device="cuda"))
    xp *= torch.exp(2 * torch.randn(x.shape, generator=g, device="cuda"))
    _check(kd.matmul_2bit(dec, x, xp), _y64(dec, x, xp))


@pytest.mark.parametrize("batch", [5, 20])
@pytest.mark.parametrize("e", [-112, -120, -130, -140, 125])
def test_rows_at_the_ends_of_the_range(kd, batch, e):  # noqa: F811
    """Rows of 2^e, subnormal ones among them, beside an ordinary row; the centres are scaled
    so that the results stay normal numbers."""
    dec, x, xp = _case(kd, 1000, 130, batch)
    dec.centres_u *= 2.0 ** (-40 if e > 0 else 40)
    dec.centres_v *= 2.0 ** (-40 if e > 0 else 40)
    x, xp = x.clamp(-4, 4), xp.clamp(-4, 4)
    x[1:] *= 2.0 ** (e // 2)
    xp[1:] *= 2.0 ** (e // 2)
    x[1:] *= 2.0 ** (e - e // 2)
    xp[1:] *= 2.0 ** (e - e // 2)
    assert torch.isfinite(x).all() and (x[1:] != 0).any(1).all()
    _check(kd.matmul_2bit(dec, x, xp), _y64(dec, x, xp))


@pytest.mark.parametrize("count", [1, 2, 64, 65, 300])
def test_infinities_of_a_row(kd, count):  # noqa: F811
    """`count` infinities in one row: infinite where their products agree in sign, else NaN;
    other rows keep their bits."""
    n = 300
    dec, x, xp = _case(kd, n, 140, 20)
    ref = kd.matmul_2bit(dec, x, xp)
    x2 = x.clone()
    at = torch.arange(count, device="cuda") * 7 % n
    x2[11, at] = float("inf")
    y = kd.matmul_2bit(dec, x2, xp)
    keep = [r for r in range(20) if r != 11]
    assert torch.equal(y[keep], ref[keep])
    sign = torch.sign(_plane(dec.codes_u, dec.centres_u, n)[:, at])
    assert (sign != 0).all()
    same = (sign == sign[:, :1]).all(1)
    assert torch.equal(y[11][same], (sign[same, 0] * float("inf")).float())
    assert torch.isnan(y[11][~same]).all()


def test_vectors_beyond_one_accumulation(kd):  # noqa: F811
    """2^16 inputs fill an accumulation: one stage into a second one, all inputs of one sign."""
    n, m, batch = 65600, 129, 17
    g = torch.Generator(device="cuda").manual_seed(1)
    codes = [torch.randint(-2 ** 31, 2 ** 31, (m, n // 16), generator=g, device="cuda").int() for _ in range(2)]
    c = torch.tensor([-1.5, -0.4, 0.4, 1.5], device="cuda").repeat(m, 1)
    dec = kd.Decomposed(*codes, c, c.clone(), None, None, None, None, None)
    x = torch.rand((batch, n), generator=g, device="cuda") + 1.0
    xp = torch.rand((batch, n), generator=g, device="cuda") + 1.0
    ref = torch.cat([_y64(dec, x[r:r + 1], xp[r:r + 1]) for r in range(batch)])
    _check(kd.matmul_2bit(dec, x, xp), ref)


@pytest.mark.parametrize("n", [300, 1000, 2112])
@pytest.mark.parametrize("batch", [5, 20])
def test_channel_with_an_unused_infinite_centre(kd, n, batch):  # noqa: F811
    """Summed plainly: the code that pads the last word has that centre and stays out; rows at an
    odd offset give the same."""
    from tests.test_gpu_fold_tc_centres import _recode
    dec, x, xp = _case(kd, n, 140, batch)
    _recode(dec.codes_u, 5, 0, 1)
    dec.centres_u[5, 0] = -float("inf")
    y = kd.matmul_2bit(dec, x, xp)
    ref = dec.centres_u.clone()
    ref[5, 0] = 0.0
    y64 = x.double() @ _plane(dec.codes_u, ref, n).t() + xp.double() @ _plane(dec.codes_v, dec.centres_v, n).t()
    assert torch.isfinite(y).all()
    assert ((y.double() - y64).abs().amax(1) <= 1e-5 * y64.abs().amax(1)).all()
    big = torch.zeros((2, batch, n + 9), device="cuda")
    big[0][:, 1:1 + n], big[1][:, 1:1 + n] = x, xp
    assert torch.equal(kd.matmul_2bit(dec, big[0][:, 1:1 + n], big[1][:, 1:1 + n]), y)
