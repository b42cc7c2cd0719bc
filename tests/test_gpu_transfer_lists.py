"""Transfers of sets small enough that their matrices travel with the launches (csrc/flora_gram.cuh, GRAM_LIST), around the number from
which a table in memory is used instead, against the oracle."""
import pytest
import torch

from paper_2402_03293_b200 import binding as fb
from tests.parity_util import oracle_transfer, rel_err

pytestmark = pytest.mark.gpu
DEV = "cuda"


# columns around a step of the product (16 to 64) and a CTA's range of them, none at all, rows around a block of the apply kernels (8 rows to 256);
# ranks of which rows are, or are not, 16-byte aligned.  fp32: products and sums in fp32, 1e-5 as elsewhere.  bf16: the rounded operands are the
# same on both sides and everything else is fp32 as well: their products are summed by the tensor core, whose truncated sums lose up to 2e-8
# of the sum per accumulation, a few hundred here at most.
@pytest.mark.parametrize("count", [2, 16, 17])
@pytest.mark.parametrize("r", [4, 33, 96])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("other_stream", [False, True])
def test_small_set_transfers(count, r, dtype, other_stream):
    shapes = [((1, 7, 64, 129, 300)[i % 5], (70, 1, 515, 0, 2049, 64)[i % 6]) for i in range(count)]
    torch.manual_seed(count * 100 + r)
    kind = torch.float32 if dtype == "f32" else torch.bfloat16
    W = [torch.zeros(n, m, dtype=kind, device=DEV) for n, m in shapes]
    src = [torch.randn(n, r, device=DEV) for n, _ in shapes]
    dst = [torch.randn(n, r, device=DEV) for n, _ in shapes]
    dst0 = [d.clone() for d in dst]
    tol = 1e-5 if dtype == "f32" else 2e-5
    a, b = fb.FloraSet(W, None, src), fb.FloraSet(None, W, dst)
    old, new = [50 + i for i in range(count)], [90 + i for i in range(count)]
    torch.cuda.synchronize()                                          # (the second stream is not ordered to the first)
    with torch.cuda.stream(torch.cuda.Stream() if other_stream else torch.cuda.current_stream()):
        b.transfer_axpby_from(a, old, new, 0.25, 0.75)
    torch.cuda.synchronize()
    for i, (n, m) in enumerate(shapes):
        want = oracle_transfer(dst0[i], src[i], m, dtype, old[i], new[i], 0.25, 0.75) if m else 0.75 * dst0[i].cpu().numpy()
        assert rel_err(dst[i].cpu().numpy(), want) <= tol, (i, n, m)
    src0 = [s.clone() for s in src]
    a.resample_transfer(old, new)                                     # in place
    for i, (n, m) in enumerate(shapes):
        want = oracle_transfer(torch.zeros_like(src0[i]), src0[i], m, dtype, old[i], new[i], 1.0, 0.0) if m else 0.0 * src0[i].cpu().numpy()
        assert rel_err(src[i].cpu().numpy(), want) <= tol, (i, n, m)
    a.close()
    b.close()
    assert fb.flora_device_status() == 0
