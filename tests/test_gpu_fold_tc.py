"""The fp32 product from the 2-bit planes for two batch rows and more (tensor cores, inputs
split into three bf16 values, codes as planes of -1, 0, 1), against the same product in
64 bits from the same codes, centres and inputs.

Sizes sit at the edges of its tiles: 128 channels, stages of 64 inputs, accumulations of 32
stages, blocks of 16 rows.

Tolerance, per row, of max |Y|: the plane sums are exact to 2^-24 of the sums themselves and
each of the at most n / 2048 + 4 fp32 operations on them rounds by 2^-24 of a value no larger
than a few max |Y|: 1e-6 covers n = 16384 four times over."""

import pytest
import torch

from paper_2609_11687_gb300 import synth
from tests.test_gpu_fold import kd  # noqa: F401  (the module's fixture)

pytestmark = pytest.mark.gpu

TOL = 1e-6


def _plane(codes, centres, n):
    q = (codes.long().unsqueeze(2) >> (2 * torch.arange(16, device=codes.device)) & 3).flatten(1)[:, :n]
    return torch.gather(centres.double(), 1, q)


def _y64(dec, x, xp):
    n = x.shape[1]
    return x.double() @ _plane(dec.codes_u, dec.centres_u, n).t() + xp.double() @ _plane(dec.codes_v, dec.centres_v, n).t()


def _case(kd, n, m, batch, kmeans=0, seed=0):  # noqa: F811
    w = synth.generate(synth.MatrixSpec("w", n, m, seed=n + m + batch, std=0.02), device="cuda")
    dec = kd.decompose(w, 4, 5, kmeans_iters=kmeans)
    g = torch.Generator(device="cuda").manual_seed(seed + batch)
    x = torch.randn((batch, n), generator=g, device="cuda")
    return dec, x, torch.randn((batch, n), generator=g, device="cuda")


@pytest.mark.parametrize("kmeans", [0, 2])  # centres symmetric about 0, and not
@pytest.mark.parametrize("n,m,batch", [
    (16, 1, 2),        # a quarter of a stage, one channel
    (64, 128, 16),     # one full stage, tile and block
    (1000, 129, 17),   # a partial code word, unaligned code rows, a second tile and block of one
    (2048, 127, 3),    # exactly one accumulation
    (4160, 130, 16),   # parts of 32 and 33 stages: an accumulation of one stage ends a part
    (1000, 19, 6),     # a partial code word and unaligned code rows in the second part
    (2112, 130, 5),    # one stage into the second
    (11008, 128, 33),  # six accumulations, three blocks
    (16384, 40, 9),
])
def test_against_64_bits(kd, n, m, batch, kmeans):  # noqa: F811
    dec, x, xp = _case(kd, n, m, batch, kmeans)
    if kmeans:
        assert not torch.equal(dec.centres_u[:, 0], -dec.centres_u[:, 3])
    y = kd.matmul_2bit(dec, x, xp)
    ref = _y64(dec, x, xp)
    err = (y.double() - ref).abs().amax(1) / ref.abs().amax(1).clamp(min=ref.abs().mean())
    assert (err <= TOL).all(), err.max().item()


def test_wide_range_of_inputs(kd):  # noqa: F811
    """Inputs over 2^-90 .. 2^60 in one row, rows of 2^-100 and of 2^100 (summed on the tensor
    cores), each against its own size."""
    n = 512
    dec, x, xp = _case(kd, n, 40, 4)
    x[1] *= torch.pow(2.0, torch.linspace(-90, 60, n, device="cuda"))
    for r, e in ((2, -100), (3, 100)):
        x[r] = x[r].clamp(-0.9, 0.9) * 2.0 ** e
        xp[r] = xp[r].clamp(-0.9, 0.9) * 2.0 ** e
    y = kd.matmul_2bit(dec, x, xp)
    ref = _y64(dec, x, xp)
    err = (y.double() - ref).abs().amax(1) / ref.abs().amax(1)
    assert (err <= TOL).all(), err


def test_non_finite_and_huge_values(kd):  # noqa: F811
    """A row with an infinity, a NaN or values that overflow a sum without its weights, and a
    channel with an infinite centre, give what fp32 products and sums give; the others keep
    their bits."""
    n, m = 300, 140
    dec, x, xp = _case(kd, n, m, 20)
    ref = kd.matmul_2bit(dec, x, xp)
    x2 = x.clone()
    x2[3, 7] = float("inf")
    x2[9, 299] = float("nan")
    x2[17, ::2] = 3e38
    x2[17, 1::2] = 0.0
    y = kd.matmul_2bit(dec, x2, xp)
    keep = [r for r in range(20) if r not in (3, 9, 17)]
    assert torch.equal(y[keep], ref[keep])
    sign = torch.sign(_plane(dec.codes_u, dec.centres_u, n)[:, 7])
    assert torch.equal(y[3], (sign * float("inf")).float())
    assert torch.isnan(y[9]).all()
    big = _y64(dec, x2[17:18], xp[17:18])[0]
    assert big.abs().max() < 3e38
    assert ((y[17].double() - big).abs() <= 1e-5 * big.abs().max()).all()
    # code 3 of channel 5 (an infinite centre), in a channel that never uses it
    d5 = _case(kd, n, m, 20)[0]
    cu = d5.codes_u.clone()
    words = cu[5].long() & 0xFFFFFFFF
    words &= ~((words & 0x55555555) & ((words >> 1) & 0x55555555))  # code 3 -> code 2
    cu[5] = torch.where(words > 0x7FFFFFFF, words - (1 << 32), words).int()
    d5.codes_u = cu
    d5.centres_u[5, 3] = float("inf")
    y = kd.matmul_2bit(d5, x, xp)
    ref5 = _y64(d5, x, xp)
    assert torch.isfinite(y).all()
    assert ((y[:, 5].double() - ref5[:, 5]).abs() <= 1e-5 * ref5.abs().max()).all()


def test_unaligned_and_strided_rows(kd):  # noqa: F811
    """Input rows at an odd element offset and stride, output rows with a stride: the bits of
    the contiguous call, nothing written beside them."""
    dec, x, xp = _case(kd, 1536, 70, 18)
    ref = kd.matmul_2bit(dec, x, xp)
    big = torch.zeros((2, 18, 1577), device="cuda")
    xs, ps = big[0][:, 1:1537], big[1][:, 1:1537]
    xs.copy_(x)
    ps.copy_(xp)
    ys = torch.full((19, 75), float("nan"), device="cuda")
    kd.matmul_2bit(dec, xs, ps, out=ys[:18, :70])
    torch.cuda.synchronize()
    assert torch.equal(ys[:18, :70], ref)
    assert torch.isnan(ys[18]).all() and torch.isnan(ys[:, 70:]).all()
