"""The TMA kernels on matrices so small that the automatic choice gives them to the kernels without TMA (flora_debug_force_path(2)):
the parity, resampling and repeatability tests over again, so that both families are compared with the oracle at ragged tiles and tails."""
import numpy as np
import pytest
import torch

from oracle import flora_oracle as orc
from paper_2402_03293_b200 import binding as fb
from paper_2402_03293_b200 import workloads as wl
from tests import test_gpu_parity as parity
from tests.parity_util import TOL, oracle_compress, rel_err

pytestmark = pytest.mark.gpu
DEV = "cuda"
ELIGIBLE = [s for s in parity.SHAPES if s[0] >= 128 and s[1] >= 64 and s[1] % 8 == 0]


@pytest.fixture(autouse=True)
def _tma():
    fb.flora_debug_force_path(2)
    yield
    fb.flora_debug_force_path(0)
    torch.cuda.synchronize()
    assert fb.flora_device_status() == 0


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("n,m,r", ELIGIBLE)
def test_single_calls(n, m, r, dtype):
    parity.test_compress_and_momentum(n, m, r, dtype, 2)
    parity.test_decompress_apply(n, m, r, dtype, 2)


@pytest.mark.parametrize("case", [c for c in range(14) if c % 3])
def test_random_sets(case):
    parity.test_random_sets_against_oracle(case)


@pytest.mark.parametrize("n,m,r", [(300, 1024, 32), (256, 4096, 128)])
def test_resampled_momentum_step(n, m, r):
    parity.test_resampled_momentum_step(n, m, r, "bf16")


def test_repeated_launches_are_bit_identical():
    parity.test_repeated_launches_are_bit_identical(768, 3072, 64)


# a set of one matrix (its transfer starts early and the compression waits for everything) and of several (whose compression starts under
# the transfer's last kernel), on compress_tc_kernel and on compress_pair_kernel, with rows and columns cut and uncut
@pytest.mark.parametrize("r", [32, 128])
@pytest.mark.parametrize("shapes", [[(384, 4104)], [(1000, 1032)], [(384, 4104), (1000, 1032), (2048, 2048)]])
def test_resampled_step_of_sets(shapes, r):
    G = [wl.gaussian_matrix(n, m, 1e-2, "bf16", 3 + i).to(DEV) for i, (n, m) in enumerate(shapes)]
    M = [torch.randn(n, r, generator=torch.Generator(device=DEV).manual_seed(i), device=DEV) for i, (n, _) in enumerate(shapes)]
    M0 = [x.clone() for x in M]
    fset = fb.FloraSet(G, None, M)
    old, new = [50 + i for i in range(len(shapes))], [60 + i for i in range(len(shapes))]
    fset.momentum_step_resampled(0.5, old, new)
    for i, (n, m) in enumerate(shapes):
        ref = wl.as_numpy(M0[i]).copy()
        orc.momentum_step_resampled(wl.as_numpy(G[i]), orc.projection(old[i], r, m, "bf16"), orc.projection(new[i], r, m, "bf16"), 0.5, ref)
        assert rel_err(M[i].cpu().numpy(), ref) <= TOL["bf16"], i
    fset.close()


# fp32 momentum on the TMA kernel: rows with one owner (read, blended and written back) and columns cut over several CTAs (scaled, then added to)
@pytest.mark.parametrize("n,m,r", [(4096, 512, 32), (256, 3104, 64), (130, 1028, 200)])
def test_fp32_momentum(n, m, r):
    G = wl.gaussian_matrix(n, m, 1e-2, "f32", 9).to(DEV)
    S0 = torch.randn(n, r, generator=torch.Generator(device=DEV).manual_seed(5), device=DEV)
    alone, member = S0.clone(), S0.clone()
    fb.flora_momentum_step(G, alone, 0.75, 34)
    fset = fb.FloraSet([G], None, [member])
    fset.momentum_step(0.75, [34])
    want = oracle_compress(G, S0, 34, a=0.25, b=0.75)
    for x in (alone, member):
        assert rel_err(x.cpu().numpy(), want) <= TOL["f32"]
    fset.close()
