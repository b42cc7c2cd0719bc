"""The kernels for fp32, unaligned and small matrices (csrc/flora_gen.cuh) at the edges of their tiles, against the oracle.

Tolerances: those of the other parity tests.  fp32: each product is exact to 2^-21 (three bf16 parts, the products left out
are below that, and 2^-24 of a sum in the 2-norm), and chains of truncated sums are kept so short that a sum over m columns is off
by less than 1.8e-8 sqrt(m): 1e-5 holds with an order of magnitude to spare at the sizes here.  The weights
carry one spacing of fp32 on top, since both sides store them rounded."""
import numpy as np
import pytest
import torch

from paper_2402_03293_b200 import binding as fb
from paper_2402_03293_b200 import workloads as wl
from tests.parity_util import TOL, oracle_compress, oracle_decompress, rel_err, values

pytestmark = pytest.mark.gpu
DEV = "cuda"


def _view(n, m, dtype, seed, offset, gap, std):
    """An n x m view that starts `offset` elements into its buffer, rows m + gap apart."""
    data = wl.gaussian_matrix(n, m, std * std, dtype, seed).to(DEV)
    buf = torch.full((offset + n * (m + gap) + 8,), 3.0, dtype=data.dtype, device=DEV)
    v = buf[offset:offset + n * (m + gap)].view(n, m + gap)[:, :m]
    v.copy_(data)
    return buf, v


# rows around one and two tiles; columns around a step (32 fp32, 64 bf16 values) and a slab; ranks around a 16-column slice,
# around where the three parts of A stop fitting one operand (80 | 96) and the largest; row groups shared by a cluster
@pytest.mark.parametrize("n,m,r", [(1, 1, 1), (127, 31, 8), (128, 33, 16), (129, 65, 17), (257, 64, 80), (300, 130, 81), (40, 1029, 96), (64, 4100, 33),
                                   (513, 257, 200), (130, 190, 256)])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("offset,gap", [(0, 0), (1, 0), (3, 5)])
def test_edges(n, m, r, dtype, offset, gap):
    gbuf, G = _view(n, m, dtype, 5, offset, gap, 0.1)
    wbuf, W = _view(n, m, dtype, 6, offset, gap, 0.02)
    _, S = _view(n, r, "f32", 7, offset, gap, 1.0)
    S0, W0 = S.clone(), W.clone()
    around = wbuf.clone()
    fb.flora_compress_accumulate(G, S, 11, r)
    assert rel_err(S.cpu().numpy(), oracle_compress(G.contiguous(), S0, 11)) <= TOL[dtype]
    S1 = S.clone()
    fb.flora_momentum_step(G, S, 0.75, 12)
    assert rel_err(S.cpu().numpy(), oracle_compress(G.contiguous(), S1, 12, a=0.25, b=0.75)) <= TOL[dtype]
    fb.flora_decompress_apply(W, S, 13, 0.03, 1.0)
    ref = oracle_decompress(W0, S.contiguous(), 13, 0.03, 1.0)
    got, want, w0 = (values(x).astype(np.float64) for x in (wl.as_numpy(W.contiguous()), ref, wl.as_numpy(W0)))
    spacing = float(np.spacing(np.float32(np.abs(want).max()))) * (1 if dtype == "f32" else 2 ** 16)
    assert np.abs(got - want).max() <= TOL[dtype] * np.abs(want - w0).max() + spacing
    W.copy_(W0)                                                       # nothing outside the view was written
    assert torch.equal(wbuf, around)
    assert fb.flora_device_status() == 0


@pytest.mark.parametrize("r", [8, 33, 128])
def test_mixed_sets(r):
    """Both dtypes, odd rows and matrices that TMA serves in one set (enough of the latter that they get their own launch)."""
    shapes = [(2048, 2304, "bf16"), (130, 515, "bf16"), (96, 200, "f32"), (10, 768, "bf16"), (300, 1000, "f32"), (50, 4099, "bf16")]
    G = [wl.gaussian_matrix(n, m, 1e-2, d, 20 + i).to(DEV) for i, (n, m, d) in enumerate(shapes)]
    W = [wl.gaussian_matrix(n, m, 4e-4, d, 40 + i).to(DEV) for i, (n, m, d) in enumerate(shapes)]
    S = [torch.randn(n, r, device=DEV) for n, _, _ in shapes]
    S0, W0 = [s.clone() for s in S], [w.clone() for w in W]
    fset = fb.FloraSet([torch.zeros_like(g) for g in G], W, S)
    fset.rebind_gradients(G)
    seeds = [fb.flora_derive_seed(3, i, 0) for i in range(len(shapes))]
    fset.momentum_step(0.5, seeds)
    for i, (n, m, d) in enumerate(shapes):
        assert rel_err(S[i].cpu().numpy(), oracle_compress(G[i], S0[i], seeds[i], a=0.5, b=0.5)) <= TOL[d], i
    fset.decompress_apply(seeds, 0.03, 1.0)
    for i, (n, m, d) in enumerate(shapes):
        ref = oracle_decompress(W0[i], S[i], seeds[i], 0.03, 1.0)
        assert rel_err(values(wl.as_numpy(W[i])), values(ref)) <= TOL[d], i
    fset.compress_overwrite(seeds)
    for i, (n, m, d) in enumerate(shapes):
        assert rel_err(S[i].cpu().numpy(), oracle_compress(G[i], torch.zeros_like(S0[i]), seeds[i])) <= TOL[d], i
    fset.zero_state()
    assert all(bool(torch.all(s == 0)) for s in S)
    fset.close()
    assert fb.flora_device_status() == 0


# fp32 matrices that the TMA compression takes (too wide or too large for the kernels above): rows and columns around a tile and a
# step, ranks around where A stops fitting one operand (128 | 129) and where two tiles share it (32 | 33), one item and several per
# accumulator set.  The bound is a third of the tolerance: hi/lo products are off by 2^-20 at most and 1.4e-7 of a sum in
# the 2-norm, and the chains of truncated sums stay below what plain fp32 sums lose, 1.8e-8 sqrt(m) in the 2-norm (2.3e-6 at 16380).
@pytest.mark.parametrize("n,m,r", [(128, 3104, 8), (257, 5000, 33), (130, 8196, 130), (385, 4100, 256), (2049, 2052, 96), (4096, 3076, 17), (129, 16380, 64),
                                   (300, 3300, 128)])
def test_fp32_through_tma(n, m, r):
    G = wl.gaussian_matrix(n, m, 1e-2, "f32", 9).to(DEV)
    S = torch.randn(n, r, device=DEV)
    S0 = S.clone()
    fb.flora_compress_accumulate(G, S, 31, r)
    A = torch.empty(r, m, device=DEV)
    fb.flora_materialize_A(A, 31)
    product = G.double() @ A.double().T
    assert ((S.double() - S0.double() - product).abs().max() / product.abs().max()).item() <= 3.3e-6 + 2.0 ** -22
    G2 = G[:, : m - 4].contiguous()
    T = S0.clone()
    fset = fb.FloraSet([torch.zeros_like(G), G2], None, [S, T])
    fset.rebind_gradients([G, G2])
    S.fill_(float("nan"))
    T.fill_(float("nan"))
    fset.compress_overwrite([32, 33])
    assert rel_err(S.cpu().numpy(), oracle_compress(G, torch.zeros_like(S), 32)) <= TOL["f32"]
    assert rel_err(T.cpu().numpy(), oracle_compress(G2, torch.zeros_like(T), 33)) <= TOL["f32"]
    S.copy_(S0)                                                       # a blend whose two parts differ: another seed, unequal weights
    T.copy_(S0)
    fset.momentum_step(0.75, [34, 35])
    assert rel_err(S.cpu().numpy(), oracle_compress(G, S0, 34, a=0.25, b=0.75)) <= TOL["f32"]
    assert rel_err(T.cpu().numpy(), oracle_compress(G2, S0, 35, a=0.25, b=0.75)) <= TOL["f32"]
    alone = S0.clone()
    fb.flora_momentum_step(G, alone, 0.75, 34)
    assert rel_err(alone.cpu().numpy(), oracle_compress(G, S0, 34, a=0.25, b=0.75)) <= TOL["f32"]
    fset.close()
    assert fb.flora_device_status() == 0


# fp32 weights that the TMA decompression takes: rows and columns around a tile, a slab and a box of 32 columns, ranks around where a
# second slab buffer stops fitting (32 | 33), with odd numbers of chunks, and the largest; next to a matrix that stays with the kernels
# above.  Per element, of sum |C| |A|: the products carry 2^-21 (lo lo left out: 2^-24; both lo cut to tf32: 2^-22 each at most), and each of the r / 8 + 2 truncated
# accumulations loses less than 2^-22 of the running sum; the store of W rounds to 2^-24.
@pytest.mark.parametrize("n,m,r", [(129, 8260, 8), (1000, 2100, 33), (4097, 1028, 1), (300, 5004, 96), (2049, 3076, 128), (8200, 164, 64), (128, 8224, 100)])
def test_fp32_weights_through_tma(n, m, r):
    W = wl.gaussian_matrix(n, m, 4e-4, "f32", 9).to(DEV)
    C = torch.randn(n, r, device=DEV)
    A = torch.empty(r, m, device=DEV)
    fb.flora_materialize_A(A, 17)
    update, size = 0.05 * (C.double() @ A.double()), 0.05 * (C.double().abs() @ A.double().abs())
    bound = size * (r / 8 + 3) * 2.0 ** -22 + (W.double().abs() + update.abs()) * 2.0 ** -24
    buf = torch.full((n, m + 4), 3.0, device=DEV)
    buf[:, :m] = W
    fb.flora_decompress_apply(buf[:, :m], C, 17, 0.05, 1.0)
    assert bool(((buf[:, :m].double() - (W.double() - update)).abs() <= bound).all()) and torch.all(buf[:, m:] == 3.0)
    small = torch.zeros(40, 70, device=DEV)
    W2 = W.clone()
    fset = fb.FloraSet(None, [W2, small], [C, torch.randn(40, r, device=DEV)])
    fset.decompress_apply([17, 18], 0.05, 1.0)
    assert bool(((W2.double() - (W.double() - update)).abs() <= bound).all()) and bool(small.abs().sum() > 0)
    fset.close()
    assert fb.flora_device_status() == 0


# Transfers: one cluster and several, with their sums stored side by side or added into one matrix (by columns and rank), ranks below,
# at and above one and two 128-row halves, ranks that TMA cannot address (33, 250), pairs of row tiles around 256, and two units per
# cluster.  Against the same product in fp64, in the Frobenius norm: with bf16 operands src and T are read as tf32, whose ten
# mantissa bits are cut off and not rounded (each value loses less than 2^-10 of itself, a product less than 2^-9, and one element of
# one row can show all of it), through the kernels without TMA and with fp32 operands everything is fp32 (1e-5 as elsewhere).
@pytest.mark.parametrize("n,m,r", [(1, 1, 4), (255, 63, 8), (257, 20000, 8), (300, 700, 33), (256, 4100, 64), (513, 2049, 128), (130, 9000, 132), (64, 515, 250),
                                   (40000, 300, 16), (385, 11008, 256)])
@pytest.mark.parametrize("operand", ["f32", "bf16"])
def test_transfer_edges(n, m, r, operand):
    dtype = torch.float32 if operand == "f32" else torch.bfloat16
    A, B = torch.empty(r, m, dtype=dtype, device=DEV), torch.empty(r, m, dtype=dtype, device=DEV)
    fb.flora_materialize_A(A, 5)
    fb.flora_materialize_A(B, 6)
    T = A.double() @ B.double().T
    tol = 2.0 ** -9 + 1e-5 if operand == "bf16" and r % 4 == 0 else 1e-5
    gen = torch.Generator(device=DEV)
    gen.manual_seed(n + m + r)
    src, old = (torch.randn(n, r, generator=gen, device=DEV) for _ in range(2))

    def size(want, a, b):
        # the errors of a sum are relative to the magnitudes of its terms; over many elements its own norm stands for them (and is the
        # sharper test), but the few elements of one row may all have cancelled
        return (want if n > 1 else a * (src.double().abs() @ T.abs()) + b * old.double().abs()).norm()
    for a, b in ((1.0, 0.0), (0.25, 0.5)):
        dst = old.clone()
        fb.flora_transfer_axpby(dst, src, m, operand, 5, 6, a, b)
        want = a * (src.double() @ T) + b * old.double()
        assert ((dst.double() - want).norm() / size(want, a, b)).item() <= tol
    # a set of two, and in place with the scratch fixed at load time
    S = [src.clone(), src[:1].clone()]
    fset = fb.FloraSet([torch.zeros(n, m, dtype=dtype, device=DEV), torch.zeros(1, m, dtype=dtype, device=DEV)], None, S)
    fset.resample_transfer([5, 7], [6, 8])
    fixed = src.clone()
    fb.flora_resample_transfer_static(fixed, m, operand, 5, 6)
    want = src.double() @ T
    assert all(((x.double() - want).norm() / size(want, 1.0, 0.0)).item() <= tol for x in (S[0], fixed))
    fset.close()
    assert fb.flora_device_status() == 0


# Rows longer than one launch may add up (36864 columns: sixteen CTAs of 72 steps), around its end and over many of them, off 16 bytes
# and, in bit-reproducible mode, on; the result stays as near to 64 bits as plain fp32 arithmetic (1.8e-8 sqrt(m) in the 2-norm; one
# chain of truncated sums over 600001 columns would lose 4e-5).
@pytest.mark.parametrize("n,m,r", [(3, 36863, 8), (130, 36865, 33), (16, 73729, 8), (5, 600001, 4), (128, 50256, 16)])
def test_long_fp32_rows(n, m, r):
    G = wl.gaussian_matrix(n, m, 1e-2, "f32", 9).to(DEV)
    A = torch.empty(r, m, device=DEV)
    fb.flora_materialize_A(A, 31)
    product = G.double() @ A.double().T
    S0 = torch.randn(n, r, generator=torch.Generator(device=DEV).manual_seed(m), device=DEV)
    fb.flora_set_deterministic(True)
    try:
        alone, again = S0.clone(), S0.clone()
        fb.flora_momentum_step(G, alone, 0.75, 31)
        fb.flora_momentum_step(G, again, 0.75, 31)
        member, other = S0.clone(), torch.ones(40, r, device=DEV)
        small = wl.gaussian_matrix(40, 300, 1e-2, "f32", 8).to(DEV)
        other0 = other.clone()
        fset = fb.FloraSet([small, G], None, [other, member])
        fset.momentum_step(0.75, [32, 31])
    finally:
        fb.flora_set_deterministic(False)
    want = 0.75 * S0.double() + 0.25 * product
    for x in (alone, member):
        assert ((x.double() - want).norm() / want.norm()).item() <= 1.8e-8 * m ** 0.5 + 2.0 ** -23
    assert torch.equal(alone, again)
    assert rel_err(other.cpu().numpy(), oracle_compress(small, other0, 32, a=0.25, b=0.75)) <= TOL["f32"]
    fset.close()
    assert fb.flora_device_status() == 0


def _special(t, seed):
    """Puts infinities, NaN and the largest numbers into some rows of t, the rest of which stays as it is; the rows that hold any."""
    n, m = t.shape
    gen = torch.Generator().manual_seed(seed)
    rows = sorted(set(torch.randint(0, n, (9,), generator=gen).tolist()) | {0, n - 1})
    for k, i in enumerate(rows):
        at = torch.randint(0, m, (3,), generator=gen).tolist() + [m - 1]
        if k % 4 == 0:
            t[i, at[0]] = float("inf")
        elif k % 4 == 1:
            t[i, at[0]], t[i, at[3]] = float("inf"), float("-inf")
        elif k % 4 == 2:
            t[i, at[1]] = float("nan")
        else:
            t[i, at[0]], t[i, at[1]] = float("-inf"), float("-inf")
    return rows


def _same(got, want, tol, what):
    """Infinities and NaN in the same places with the same signs; the numbers within tol of the largest."""
    got, want = got.double(), want.double()
    fin = torch.isfinite(want)
    assert torch.equal(torch.isnan(got), torch.isnan(want)) and torch.equal(got[torch.isinf(want)], want[torch.isinf(want)]), what
    assert bool((got[fin] - want[fin]).abs().max() <= tol * want[fin].abs().max()), what


# Infinities and NaN come out as plain arithmetic gives them wherever fp32 values are multiplied in parts: fp32 gradients in the kernels
# without TMA (split over a cluster or not, off 16 bytes or on) and with it (one item or several per row, one operand or two, a
# cluster), sketches in both decompressions and for bf16 weights of the kernels without TMA.
@pytest.mark.parametrize("n,m,r,offset", [(200, 300, 8, 0), (130, 1029, 33, 1), (64, 4100, 96, 0), (300, 5000, 17, 0), (257, 4100, 130, 0), (2049, 2052, 64, 0)])
def test_infinities_in_gradients(n, m, r, offset):
    _, G = _view(n, m, "f32", 3, offset, 0, 0.1)
    _special(G, 1)
    A = torch.empty(r, m, device=DEV)
    fb.flora_materialize_A(A, 31)
    product = torch.stack([(G.double() * A[j].double()).sum(1) for j in range(r)], 1)       # (no zeros are multiplied in)
    S = torch.randn(n, r, generator=torch.Generator(device=DEV).manual_seed(5), device=DEV)
    S0 = S.clone()
    fb.flora_compress_accumulate(G, S, 31, r)
    _same(S, S0.double() + product, 1e-5, "add")
    S.fill_(float("nan"))
    fb.flora_momentum_step(G, S, 0.0, 31)
    _same(S, product, 1e-5, "overwrite")
    T = S0.clone()
    fset = fb.FloraSet([torch.zeros_like(G), torch.zeros_like(G)], None, [T, S])
    fset.rebind_gradients([G, G])
    fset.momentum_step(0.75, [31, 32])
    _same(T, 0.75 * S0.double() + 0.25 * product, 1e-5, "momentum of a set")
    fset.close()


@pytest.mark.parametrize("n,m,r,dtype", [(200, 300, 8, "f32"), (130, 1029, 96, "f32"), (2049, 3076, 64, "f32"), (600, 5004, 128, "f32"), (130, 1029, 33, "bf16"),
                                         (300, 384, 16, "bf16"), (2049, 3080, 32, "bf16")])
def test_infinities_in_sketches(n, m, r, dtype):
    C = torch.randn(n, r, generator=torch.Generator(device=DEV).manual_seed(6), device=DEV)
    rows = _special(C, 2)
    if dtype == "f32" and r >= 64:                                    # (|A| < 5.8 / sqrt(r): the sum stays finite)
        C[rows[1]] = 1e-3
        C[rows[1], r - 1] = 3.4028234e38                              # rounds to infinity in tf32
    A = torch.empty(r, m, device=DEV, dtype=wl.torch_dtype(dtype))
    fb.flora_materialize_A(A, 17)
    W = wl.gaussian_matrix(n, m, 4e-4, dtype, 9).to(DEV)
    update = torch.zeros(n, m, device=DEV, dtype=torch.float64)
    for j in range(r):
        update += C[:, j:j + 1].double() * A[j].double()
    want = W.double() - 1e-3 * update
    W2 = W.clone()
    fb.flora_decompress_apply(W, C, 17, 1e-3, 1.0)
    fset = fb.FloraSet(None, [W2, W2.clone()], [C, C])
    fset.decompress_apply([17, 18], 1e-3, 1.0)
    big = want.abs() > 1e30
    for x in (W, W2):
        _same(torch.where(big, 0.0, x.double()), torch.where(big, 0.0, want), 1e-5 if dtype == "f32" else 4e-3, "numbers")
        _same(torch.where(big, x.double(), 0.0), torch.where(big, want, 0.0), 1e-5 if dtype == "f32" else 4e-3, "large")
    fset.close()
    assert fb.flora_device_status() == 0


# A set with matrices that TMA cannot address: its transfer is computed in fp32 throughout (as tf32 the sketches would be off by 8e-4).
@pytest.mark.parametrize("r", [32, 64])
def test_transfers_of_mixed_sets_stay_in_fp32(r):
    shapes = [(130, 70), (1000, 515), (257, 4097), (768, 768), (48, 3072)]
    src = [torch.randn(n, r, generator=torch.Generator(device=DEV).manual_seed(i), device=DEV) for i, (n, _) in enumerate(shapes)]
    dst = [torch.randn(n, r, generator=torch.Generator(device=DEV).manual_seed(9 + i), device=DEV) for i, (n, _) in enumerate(shapes)]
    dst0 = [x.clone() for x in dst]
    G = [torch.zeros(n, m, device=DEV, dtype=torch.bfloat16) for n, m in shapes]
    acc, mom = fb.FloraSet(G, None, src), fb.FloraSet(None, [g.clone() for g in G], dst)
    mom.transfer_axpby_from(acc, [1, 2, 3, 4, 5], [11, 12, 13, 14, 15], 0.25, 0.5)
    for i, (n, m) in enumerate(shapes):
        A, B = torch.empty(r, m, dtype=torch.bfloat16, device=DEV), torch.empty(r, m, dtype=torch.bfloat16, device=DEV)
        fb.flora_materialize_A(A, 1 + i)
        fb.flora_materialize_A(B, 11 + i)
        want = 0.25 * (src[i].double() @ (A.double() @ B.double().T)) + 0.5 * dst0[i].double()
        assert ((dst[i].double() - want).norm() / want.norm()).item() <= 1e-5, i
    acc.close()
    mom.close()
