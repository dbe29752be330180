"""The 16-bit product from the 2-bit planes for short vectors and many rows (tcgen05): how many
additions the tensor core chains, seen in the error against 64 bits on the same 16-bit inputs
and centres.

Tolerance, 2-norm relative to the result's: a chain of s = max(8, n / 32) steps, each cut off by
half of 2^-23 of the running sum on average and all towards zero; the running sum's size after k
of s steps is sqrt(k / s) of the last (2/3 on average), so 2/3 s 2^-24, and 2 2^-24 for the fp32
sums of the chains."""

import pytest
import torch

from paper_2609_11687_gb300 import synth
from tests.test_gpu_fold import kd  # noqa: F401  (the module's fixture)
from tests.test_gpu_fold_tc import _plane

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [torch.float16, torch.bfloat16])
@pytest.mark.parametrize("n", [256, 300, 512, 768])
@pytest.mark.parametrize("batch", [65, 129, 300])
def test_error_of_short_vectors(kd, n, batch, dtype):  # noqa: F811
    w = synth.generate(synth.MatrixSpec("w", n, 300, seed=n, std=0.02), device="cuda")
    dec = kd.decompose(w, 4, 5)
    g = torch.Generator(device="cuda").manual_seed(batch)
    x, xp = (torch.randn((batch, n), generator=g, device="cuda").to(dtype) for _ in range(2))
    y = kd.matmul_2bit_f16(dec, x, xp).double()
    ref = x.double() @ _plane(dec.codes_u, dec.centres_u.to(dtype), n).t() \
        + xp.double() @ _plane(dec.codes_v, dec.centres_v.to(dtype), n).t()
    tol = (max(8, n / 32) * 2 / 3 + 2) * 2.0 ** -24
    assert (y - ref).norm() <= tol * ref.norm(), ((y - ref).norm() / ref.norm() / tol).item()


@pytest.mark.parametrize("n", [128, 300, 640])
@pytest.mark.parametrize("batch", [70, 140])
def test_rows_that_tma_cannot_read(kd, n, batch):  # noqa: F811
    """Short accumulations with the B tiles filled by the threads: the bits of aligned rows."""
    dec = kd.decompose(synth.generate(synth.MatrixSpec("w", n, 150, seed=n, std=0.02), device="cuda"), 4, 5)
    g = torch.Generator(device="cuda").manual_seed(batch)
    x, xp = (torch.randn((batch, n), generator=g, device="cuda").half() for _ in range(2))
    pad = -n % 8  # aligned rows for the reference call
    big = torch.zeros((2, batch, n + pad + 9), device="cuda", dtype=torch.float16)
    al = torch.zeros((2, batch, n + pad), device="cuda", dtype=torch.float16)
    for i, t in enumerate((x, xp)):
        big[i][:, 1:1 + n] = t
        al[i][:, :n] = t
    ref = kd.matmul_2bit_f16(dec, al[0][:, :n], al[1][:, :n])
    assert torch.equal(kd.matmul_2bit_f16(dec, big[0][:, 1:1 + n], big[1][:, 1:1 + n]), ref)
