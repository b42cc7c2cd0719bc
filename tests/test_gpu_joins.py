"""Compressions whose columns are shared by several CTAs (csrc/flora_gen.cuh), in bit-reproducible mode and without: sums sent to the CTA that owns a row, or stored in
scratch and added up by a kernel behind; row counts around a tile and a CTA's share of its rows, columns around a step, ranks on both sides of the 16-byte
accesses.  The sums are added in a fixed order: the same bits from run to run in either mode.

Tolerance against 64 bits, in the 2-norm: 1.8e-8 sqrt(m) for the products and their sums (what plain fp32 arithmetic is off by), and 3e-8 for the one rounding
of the sketch (2^-25 of its values on average)."""
import pytest
import torch

from paper_2402_03293_b200 import binding as fb
from paper_2402_03293_b200 import workloads as wl

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.fixture(autouse=True)
def _ordered_off():
    yield
    fb.flora_set_deterministic(False)
    assert fb.flora_device_status() == 0


@pytest.mark.parametrize("n,m,r", [(1, 65, 4), (7, 1000, 17), (127, 4100, 64), (129, 520, 255), (300, 33, 8), (1000, 4097, 64), (770, 2304, 16)])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("ordered", [False, True])
def test_split_sums(n, m, r, dtype, ordered):
    fb.flora_set_deterministic(ordered)
    G = wl.gaussian_matrix(n, m, 1e-2, dtype, 3).to(DEV)
    A = torch.empty(r, m, dtype=G.dtype, device=DEV)
    fb.flora_materialize_A(A, 21)
    product = G.double() @ A.double().T
    bound = 1.8e-8 * max(m, 64) ** 0.5 + 3e-8

    def off(S, want):
        return ((S.double() - want).norm() / want.norm()).item()

    S0 = torch.randn(n, r, device=DEV)
    S = S0.clone()
    fb.flora_compress_accumulate(G, S, 21, r)
    assert off(S, S0.double() + product) <= bound
    S = S0.clone()
    fb.flora_momentum_step(G, S, 0.75, 21)
    assert off(S, 0.75 * S0.double() + 0.25 * product) <= bound
    again = S0.clone()
    fb.flora_momentum_step(G, again, 0.75, 21)
    assert torch.equal(S, again)
    S = torch.full((n, r), float("nan"), device=DEV)                  # (nothing of it may be read)
    fb.flora_momentum_step(G, S, 0.0, 21)
    assert off(S, product) <= bound
    other = torch.full((n + 5, r), 2.0, device=DEV)                   # a member of a set beside a matrix of another height
    small = wl.gaussian_matrix(n + 5, 70, 1e-2, dtype, 4).to(DEV)
    S = S0.clone()
    fset = fb.FloraSet([small, G], None, [other, S])
    fset.momentum_step(0.75, [22, 21])
    fset.compress_accumulate([22, 21])
    assert off(S, 0.75 * S0.double() + 1.25 * product) <= bound
    again = S.clone()
    S.copy_(S0)
    fset.momentum_step(0.75, [22, 21])
    fset.compress_accumulate([22, 21])
    assert torch.equal(S, again)
    fset.close()
