"""The products recorded in a CUDA graph (the fp32 one's two launches overlap by a programmatic
dependency) and run on two streams at once: the bits of plain calls."""

import pytest
import torch

from tests.test_gpu_fold import kd  # noqa: F401  (the module's fixture)
from tests.test_gpu_fold_tc import _case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("half,batch", [(False, 2), (False, 16), (False, 40), (True, 4), (True, 33), (True, 300)])
def test_replayed_graph(kd, half, batch):  # noqa: F811
    dec, x, xp = _case(kd, 768, 4096, batch)
    d2, x2, xp2 = _case(kd, 4096, 1100, batch)
    args = [x, x2, xp, xp2]
    if half:
        args = [a.half() for a in args]
    call = kd.matmul_2bit_f16_batch if half else kd.matmul_2bit_batch
    ys = [torch.empty((batch, 4096), device="cuda"), torch.empty((batch, 1100), device="cuda")]
    ref = [y.clone() for y in call([dec, d2], args[:2], args[2:])]
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        call([dec, d2], args[:2], args[2:], outs=ys)
    for _ in range(3):
        for y in ys:
            y.fill_(float("nan"))
        g.replay()
        assert all(torch.equal(y, r) for y, r in zip(ys, ref))
    args[0].mul_(0.5)
    args[2].mul_(0.5)
    ref2 = call([dec, d2], args[:2], args[2:])
    g.replay()
    assert all(torch.equal(y, r) for y, r in zip(ys, ref2))


def test_two_streams(kd):  # noqa: F811
    """Both tensor-core kernels on the same SMs, many calls in flight on each stream."""
    d1, x1, xp1 = _case(kd, 4096, 4096, 40)
    d2, x2, xp2 = _case(kd, 4096, 4096, 100)
    x2, xp2 = x2.half(), xp2.half()
    r1, r2 = kd.matmul_2bit(d1, x1, xp1).clone(), kd.matmul_2bit_f16(d2, x2, xp2).clone()
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    y1 = [torch.empty_like(r1) for _ in range(20)]
    y2 = [torch.empty_like(r2) for _ in range(20)]
    for a, b in zip(y1, y2):
        kd.matmul_2bit(d1, x1, xp1, out=a, stream=s1)
        kd.matmul_2bit_f16(d2, x2, xp2, out=b, stream=s2)
    torch.cuda.synchronize()
    assert all(torch.equal(a, r1) for a in y1) and all(torch.equal(b, r2) for b in y2)
