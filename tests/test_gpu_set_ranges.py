"""Column ranges that the CTAs of a set's compression take where one matrix is much wider than it is tall (csrc/flora_gen_host.cuh)."""
import pytest
import torch

from paper_2402_03293_b200 import binding as fb

pytestmark = pytest.mark.gpu
DEV = "cuda"


# From a few steps of 64 columns to half a million of them, where part * steps leaves 32 bits if a row is cut into too many parts.  The tensor core
# truncates its sums, by 2e-8 of the running sum for each of a part's 4 * steps / 64 accumulations (measured), 6.2e-4 for the widest; a range left out or
# taken twice shows as the square root of its share of the columns.
@pytest.mark.parametrize("m", [4097, 70001, 1000003, 31765017])
def test_wide_member(m):
    torch.manual_seed(m)
    r = 8
    G = [torch.randn(1, m, device=DEV).bfloat16(), torch.randn(130, 70, device=DEV).bfloat16()]
    S = [torch.randn(g.shape[0], r, device=DEV) for g in G]
    S0 = [s.clone() for s in S]
    fset = fb.FloraSet(G, None, S)
    fset.compress_accumulate([5, 6])
    for i, g in enumerate(G):
        A = torch.empty(r, g.shape[1], dtype=torch.bfloat16, device=DEV)
        fb.flora_materialize_A(A, 5 + i)
        want = sum(x.double() @ a.double().T for x, a in zip(g.split(1 << 20, 1), A.split(1 << 20, 1)))
        assert ((S[i].double() - S0[i].double() - want).norm() / want.norm()).item() <= 2e-6 + 4 * (g.shape[1] / 64 / 64 + 1) * 2e-8, i
    fset.close()
    assert fb.flora_device_status() == 0
