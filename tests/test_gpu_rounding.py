"""A step rounds what is added to a sketch into it once, however many CTAs share the sums (csrc/flora_fold.cuh), against 64-bit arithmetic.

Bound in the 2-norm: 2^-25 of the result's values for that one rounding (2.5e-8 on average over their mantissas, measured 2.2e-8 to 2.6e-8), 3e-8 here, and
what the product's own sums are off by.  Every part rounded in by itself shows as the square root of their number."""
import pytest
import torch

from paper_2402_03293_b200 import binding as fb
from paper_2402_03293_b200 import workloads as wl

pytestmark = pytest.mark.gpu
DEV = "cuda"


def _sketch(n, r, offset):
    return torch.zeros(offset + n * r, device=DEV)[offset:].view(n, r)


def _projection(G, r, seed):
    A = torch.empty(r, G.shape[1], dtype=G.dtype, device=DEV)
    fb.flora_materialize_A(A, seed)
    return A.double()


def _check(states, gradients, calls, ratio, sums):
    """calls: (beta or None, function); sums: error that the products' sums may have, of a product, by its columns."""
    products = [G.double() @ _projection(G, S.shape[1], 40 + i).T for i, (G, S) in enumerate(zip(gradients, states))]
    start = [(torch.randn_like(S) * (ratio * p.norm().item() / p.numel() ** 0.5)) for S, p in zip(states, products)]
    for beta, call in calls:
        for S, s in zip(states, start):
            S.copy_(s)
        call()
        a, b = (1.0, 1.0) if beta is None else (1.0 - torch.tensor(beta).item(), torch.tensor(beta).item())
        for i, (S, s, p) in enumerate(zip(states, start, products)):
            want = b * s.double() + a * p
            m = gradients[i].shape[1]
            launches = -(-m // 36864) if gradients[i].dtype == torch.float32 else 1        # (each takes so many columns of an fp32 matrix at most)
            assert ((S.double() - want).norm() <= 3e-8 * launches ** 0.5 * want.norm() + sums(m) * a * p.norm()).item(), (beta, ratio, i)
    assert fb.flora_device_status() == 0


def _single(n, m, r, dtype, offset, ratio, sums):
    G, S = wl.gaussian_matrix(n, m, 1e-2, dtype, 3).to(DEV), _sketch(n, r, offset)
    _check([S], [G], [(None, lambda: fb.flora_compress_accumulate(G, S, 40, r)), (0.75, lambda: fb.flora_momentum_step(G, S, 0.75, 40))], ratio, sums)


def _set(shapes, r, dtype, offset, ratio, sums):
    G = [wl.gaussian_matrix(n, m, 1e-2, dtype, 3 + i).to(DEV) for i, (n, m) in enumerate(shapes)]
    S = [_sketch(n, r, offset) for n, _ in shapes]
    fset, seeds = fb.FloraSet(G, None, S), [40 + i for i in range(len(shapes))]
    _check(S, G, [(None, lambda: fset.compress_accumulate(seeds)), (0.75, lambda: fset.momentum_step(0.75, seeds))], ratio, sums)
    fset.close()


# Sketches that TMA cannot address, of matrices that it can: 7e-8 of a sum lost per step of 64 columns of a CTA's part by the tensor core, which is at most what the
# general kernels would lose (8 parts or more of the single matrices, two of the set's).
@pytest.mark.parametrize("ratio", [1, 1000])
@pytest.mark.parametrize("n,m,r,offset", [(4096, 11008, 7, 0), (2048, 4096, 128, 1), (1224, 4896, 255, 0)])
def test_sketches_that_tma_cannot_address(n, m, r, offset, ratio):
    _single(n, m, r, "bf16", offset, ratio, lambda m: 7e-8 * m / 64 / 8)


@pytest.mark.parametrize("ratio", [1, 1000])
@pytest.mark.parametrize("r,offset", [(31, 0), (101, 0), (32, 1)])
def test_sets_of_such_sketches(r, offset, ratio):
    _set([(1192, 3576), (1192, 1192), (1192, 4768), (4768, 1192)] * 2, r, "bf16", offset, ratio, lambda m: 7e-8 * 4768 / 64 / 2)


# The general kernels, by clusters and by single CTAs whose sums a second kernel adds up: what plain fp32 sums are off by (fp32), or 7e-8 per step of a CTA's part (bf16:
# four parts at least where there are more than 512 columns, two in a set).  One row group and many, rows and ranks off the pieces of four, fp32 rows of two launches.
def _general(dtype, parts):
    return (lambda m: 1.8e-8 * max(m, 64) ** 0.5) if dtype == "f32" else (lambda m: 7e-8 * (m / 64 / (parts if m > 512 else 1) + 1))


@pytest.mark.parametrize("ratio", [1, 1000])
@pytest.mark.parametrize("n,m,r,dtype", [(512, 512, 8, "f32"), (300, 700, 33, "f32"), (3000, 5001, 18, "f32"), (3456, 145, 256, "f32"), (200, 40001, 24, "f32"),
                                         (2048, 2048, 64, "f32"), (256, 384, 32, "bf16"), (95, 3057, 17, "bf16"), (1000, 4097, 64, "bf16"), (2048, 2048, 32, "bf16"),
                                         (129, 520, 255, "bf16"), (3000, 2001, 128, "bf16")])
def test_general_kernels(n, m, r, dtype, ratio):
    _single(n, m, r, dtype, 0, ratio, _general(dtype, 4))


@pytest.mark.parametrize("ratio", [1, 1000])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("r", [8, 33, 255])
@pytest.mark.parametrize("shapes", [[(130, 70), (1000, 515), (257, 4097), (128, 64), (4000, 129), (768, 768), (10, 768), (50, 3072)], [(127, 4100), (64, 40001)]])
def test_sets_of_general_kernels(shapes, r, dtype, ratio):
    _set(shapes, r, dtype, 0, ratio, _general(dtype, 2))
