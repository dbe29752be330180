"""Which kernel a matrix of the 16-bit product takes for short vectors of many channels, at both
sides of each line: against 64 bits on the same 16-bit inputs and centres, and the same bits
alone and in a call with matrices of the other side.

Tolerance, per row, of max |Y|: 1e-5, that of test_gpu_fold16."""

import pytest
import torch

from tests.test_gpu_fold import TOL, kd  # noqa: F401  (the module's fixture)
from tests.test_gpu_fold_tc import _case, _plane

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [torch.float16, torch.bfloat16])
@pytest.mark.parametrize("n,m,batch", [
    (1024, 8192, 1), (1024, 8193, 8), (1024, 8192, 9), (1000, 8200, 16), (16, 8192, 13), (1024, 8191, 12),
    (1029, 8192, 5), (1040, 8192, 16), (768, 8192, 17), (256, 16384, 17), (256, 16390, 32), (250, 16385, 25),
    (256, 16383, 20), (260, 16384, 20), (256, 16384, 33)])
def test_both_sides(kd, n, m, batch, dtype):  # noqa: F811
    dec, x, xp = _case(kd, n, m, batch)
    x, xp = x.to(dtype), xp.to(dtype)
    y = kd.matmul_2bit_f16(dec, x, xp)
    ref = x.double() @ _plane(dec.codes_u, dec.centres_u.to(dtype), n).t() \
        + xp.double() @ _plane(dec.codes_v, dec.centres_v.to(dtype), n).t()
    assert ((y.double() - ref).abs().amax(1) <= TOL * ref.abs().amax(1)).all()
    big = torch.zeros((2, batch, n + 41), device="cuda", dtype=dtype)  # rows at an odd offset
    xs, ps = big[0][:, 3:3 + n], big[1][:, 3:3 + n]
    xs.copy_(x)
    ps.copy_(xp)
    d2, x2, xp2 = _case(kd, 2048, 100, batch)
    x2, xp2 = x2.to(dtype), xp2.to(dtype)
    ys = torch.full((batch + 1, m + 9), float("nan"), device="cuda")
    y2 = torch.empty((batch, 100), device="cuda")
    kd.matmul_2bit_f16_batch([d2, dec], [x2, xs], [xp2, ps], outs=[y2, ys[:batch, :m]])
    assert torch.equal(ys[:batch, :m], y) and torch.equal(y2, kd.matmul_2bit_f16(d2, x2, xp2))
    assert torch.isnan(ys[batch]).all() and torch.isnan(ys[:, m:]).all()
