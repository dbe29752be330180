"""The 16-bit product from the 2-bit planes for more than 8 batch rows (tcgen05), against
the fp64 oracle on the same 16-bit inputs and centres.

Sizes sit at the edges of its tiles: 128 channels, 128 inputs per unit, accumulations of 8
units, clusters of four CTAs up to 64 rows and of two up to 128, row blocks of 256.

Tolerance (of test_gpu_fold16): 1e-5 of max |Y| per row, times sqrt(n / 4096) beyond n =
4096.  A TMEM accumulation is 64 steps of at most 2^-23 of its running sum each, 7.6e-6 of
that partial sum, and the partial sums are added in fp32."""

import numpy as np
import pytest
import torch

from tests.test_gpu_fold16 import _exact, kd  # noqa: F401  (the module's fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,m,batch,bf16", [
    (100, 30, 9, True),        # the fewest rows, one unit per plane
    (4096, 128, 16, False),    # a full block of 16 rows
    (16, 1, 17, False),        # half a unit, three of the four CTAs of a cluster idle
    (128, 128, 64, True),      # one unit per plane, one full tile
    (1000, 129, 65, False),    # a partial code word, unaligned code rows, a second tile of one channel
    (1152, 127, 128, True),    # 18 units over two CTAs: one unit into the second accumulation
    (2048, 130, 129, False),   # one CTA per tile, 32 units
    (4096, 256, 257, True),    # two row blocks of 144 (the last of 113)
    (11008, 128, 33, False),   # 172 units, accumulations of every CTA past two buffers
    (768, 40, 600, True),      # three row blocks
])
def test_exact_inputs(kd, n, m, batch, bf16):  # noqa: F811
    g = torch.Generator(device="cuda").manual_seed(n + m + batch)
    w = (torch.randn((m, n), generator=g, device="cuda") * 0.02).half()
    _exact(kd, w, 5, batch, iters=4, gen_seed=batch, bf16=bf16)


@pytest.mark.parametrize("batch", [20, 100, 300])
def test_unaligned_rows_and_batched_calls_give_the_same_bits(kd, batch):  # noqa: F811
    """Rows that TMA cannot read (an odd element offset; an odd stride) are filled by the
    threads: the same bits as the aligned rows, alone and in one call with them; nothing
    past m or past the batch is written."""
    g = torch.Generator(device="cuda").manual_seed(batch)
    m, n = 150, 1536
    w = (torch.randn((m, n), generator=g, device="cuda") * 0.02).half()
    dec = kd.decompose(w, 4, 8)
    x16 = torch.randn((batch, n), generator=g, device="cuda").half()
    xp16 = kd.apply_p(x16.float(), 8).half()
    ref = kd.matmul_2bit_f16(dec, x16, xp16)
    big = torch.zeros((2, batch + 1, n + 41), device="cuda", dtype=torch.float16)
    xs, ps = big[0][:batch, 3:3 + n], big[1][:batch, 3:3 + n]
    xs.copy_(x16)
    ps.copy_(xp16)
    ys = torch.full((batch + 1, m + 9), float("nan"), device="cuda")
    y1 = ys[:batch, :m]
    a, b = kd.matmul_2bit_f16_batch([dec, dec], [x16, xs], [xp16, ps], outs=[torch.empty_like(ref), y1])
    torch.cuda.synchronize()
    assert torch.equal(a, ref) and torch.equal(b, ref)
    assert torch.isnan(ys[batch:]).all() and torch.isnan(ys[:, m:]).all()


def test_non_finite_rows_stay_apart(kd):  # noqa: F811
    """Infinities and NaN in one batch row reach that row's outputs alone."""
    g = torch.Generator(device="cuda").manual_seed(3)
    w = (torch.randn((140, 512), generator=g, device="cuda") * 0.02).half()
    dec = kd.decompose(w, 4, 2)
    x = torch.randn((40, 512), generator=g, device="cuda").half()
    xp = kd.apply_p(x.float(), 2).half()
    ref = kd.matmul_2bit_f16(dec, x, xp)
    x2 = x.clone()
    x2[7, 5] = float("inf")
    x2[30, 511] = float("nan")
    y = kd.matmul_2bit_f16(dec, x2, xp)
    torch.cuda.synchronize()
    keep = np.setdiff1d(np.arange(40), [7, 30])
    assert torch.equal(y[keep], ref[keep])
    assert not torch.isfinite(y[7]).any() and torch.isnan(y[30]).all()
