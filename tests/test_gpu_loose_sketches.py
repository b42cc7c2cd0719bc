"""bf16 matrices that TMA can address with sketches that it cannot: ranks that are no multiple of four, strides and bases off 16 bytes, on
the TMA kernels (flora_debug_force_path(2) takes them at these sizes, too), against the oracle."""
import numpy as np
import pytest
import torch

from paper_2402_03293_b200 import binding as fb
from paper_2402_03293_b200 import workloads as wl
from tests.parity_util import TOL, oracle_compress, oracle_decompress, rel_err, values

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.fixture(autouse=True)
def _tma():
    fb.flora_debug_force_path(2)
    yield
    fb.flora_debug_force_path(0)
    torch.cuda.synchronize()
    assert fb.flora_device_status() == 0


def _sketch(n, r, offset, gap, seed, fill=None):
    """A sketch that starts `offset` floats into its buffer, rows r + gap apart, and the buffer (whose other values may not change)."""
    buf = torch.full((offset + n * (r + gap) + 8,), 3.0, device=DEV)
    S = buf[offset:offset + n * (r + gap)].view(n, r + gap)[:, :r]
    S.copy_(torch.randn(n, r, generator=torch.Generator().manual_seed(seed)) if fill is None else torch.full((n, r), fill))
    return buf, S


def _weights_match(W, W0, S, seed, lr):
    ref = oracle_decompress(W0, S.contiguous(), seed, lr, 1.0)
    got, want, w0 = (values(x).astype(np.float64) for x in (wl.as_numpy(W), ref, wl.as_numpy(W0)))
    spacing = float(np.spacing(np.float32(np.abs(want).max()))) * 2 ** 16          # (both sides store W rounded to bf16)
    assert np.abs(got - want).max() <= TOL["bf16"] * np.abs(want - w0).max() + spacing


# ranks around the chunks of 32 columns that are written out and of 64 that are multiplied, in both compression kernels (to 64, above) and
# both decompression kernels (to 128, above); rows cut and uncut
@pytest.mark.parametrize("n,m", [(128, 64), (300, 1000), (1100, 520)])
@pytest.mark.parametrize("r,offset,gap", [(1, 0, 0), (7, 0, 0), (9, 1, 0), (17, 0, 0), (31, 0, 2), (32, 1, 0), (33, 0, 0), (63, 0, 0), (64, 2, 0), (65, 0, 0), (101, 0, 3), (129, 0, 0),
                                          (192, 3, 0), (255, 0, 0)])
def test_single_calls(n, m, r, offset, gap):
    G, W = wl.gaussian_matrix(n, m, 1e-2, "bf16", 5).to(DEV), wl.gaussian_matrix(n, m, 4e-4, "bf16", 6).to(DEV)
    W0 = W.clone()
    buf, S = _sketch(n, r, offset, gap, 7)
    outside = buf.clone()
    S0 = S.clone()
    fb.flora_compress_accumulate(G, S, 11, r)
    assert rel_err(S.cpu().numpy(), oracle_compress(G, S0.contiguous(), 11)) <= TOL["f32"]
    S0 = S.clone()
    fb.flora_momentum_step(G, S, 0.75, 12)
    assert rel_err(S.cpu().numpy(), oracle_compress(G, S0.contiguous(), 12, a=0.25, b=0.75)) <= TOL["f32"]
    S.fill_(float("nan"))
    fb.flora_momentum_step(G, S, 0.0, 13)
    assert rel_err(S.cpu().numpy(), oracle_compress(G, torch.zeros(n, r), 13)) <= TOL["f32"]
    fb.flora_decompress_apply(W, S, 14, 0.03, 1.0)
    _weights_match(W, W0, S, 14, 0.03)
    outside[offset:offset + n * (r + gap)].view(n, r + gap)[:, :r].copy_(S)
    assert torch.equal(buf, outside)                                  # nothing beside the sketch was written


@pytest.mark.parametrize("r", [12, 45, 130])
def test_sets(r):
    """Sketches that TMA can and cannot address in one set (strides of r + 1 for every other one)."""
    shapes = [(256, 512), (130, 200), (2100, 1024), (384, 3000)]
    G = [wl.gaussian_matrix(n, m, 1e-2, "bf16", 20 + i).to(DEV) for i, (n, m) in enumerate(shapes)]
    W = [wl.gaussian_matrix(n, m, 4e-4, "bf16", 40 + i).to(DEV) for i, (n, m) in enumerate(shapes)]
    S = [_sketch(n, r, 0, i % 2, 60 + i)[1] for i, (n, _) in enumerate(shapes)]
    seeds = [70 + i for i in range(len(shapes))]
    fset = fb.FloraSet(G, W, S)
    for beta in (None, 0.75, 0.0):
        S0 = [s.clone() for s in S]
        if beta is None:
            fset.compress_accumulate(seeds)
        else:
            fset.momentum_step(beta, seeds)
        for i in range(len(shapes)):
            want = oracle_compress(G[i], S0[i], seeds[i]) if beta is None else oracle_compress(G[i], S0[i], seeds[i], a=1.0 - beta, b=beta)
            assert rel_err(S[i].cpu().numpy(), want) <= TOL["f32"], (beta, i)
    W0 = [w.clone() for w in W]
    fset.decompress_apply(seeds, 0.03, 1.0)
    for i in range(len(shapes)):
        _weights_match(W[i], W0[i], S[i], seeds[i], 0.03)
    S[0].fill_(float("inf"))                                          # parts of an infinity: the sign of the projection decides, no NaN
    S[1].zero_()
    fset.decompress_apply(seeds, 0.03, 1.0)
    assert not torch.isfinite(W[0].float()).any()
    assert torch.isfinite(W[1].float()).all()
    fset.close()


def test_first_calls_of_a_shape_inside_a_graph():
    """Nothing is planned for such sketches while a stream is being recorded (and a replay reads what the buffers hold by then)."""
    n, m, r = 4112, 4104, 75                                          # (a shape of its own: no plan of another test)
    G, W = wl.gaussian_matrix(n, m, 1e-2, "bf16", 1).to(DEV), wl.gaussian_matrix(n, m, 4e-4, "bf16", 2).to(DEV)
    S = torch.zeros(n, r, device=DEV)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        fb.flora_momentum_step(G, S, 0.0, 3)
        fb.flora_compress_accumulate(G, S, 3, r)
        fb.flora_decompress_apply(W, S, 3, 0.01, 0.5)
    W0, G2 = W.clone(), wl.gaussian_matrix(n, m, 1e-2, "bf16", 4).to(DEV)
    G.copy_(G2)
    graph.replay()
    rows = np.arange(0, n, 257)
    want = 2.0 * oracle_compress(G2[rows].contiguous(), torch.zeros(len(rows), r), 3)
    assert rel_err(S[rows].cpu().numpy(), want) <= TOL["f32"]
    wref = oracle_decompress(W0[rows].contiguous(), S[rows].contiguous(), 3, 0.01, 0.5)
    assert rel_err(values(wl.as_numpy(W[rows].contiguous())), values(wref)) <= TOL["bf16"]
    del graph


@pytest.mark.parametrize("path", [0, 2])
def test_one_odd_sketch_among_others(path):
    """It takes its own matrix to other kernels, and only that one: the others' results are those of a set without it, bit for bit."""
    fb.flora_debug_force_path(path)
    r, shapes = 64, [(2048, 1024), (1000, 2048), (2048, 1024), (512, 2048)]
    G = [wl.gaussian_matrix(n, m, 1e-2, "bf16", 80 + i).to(DEV) for i, (n, m) in enumerate(shapes)]
    W0 = [wl.gaussian_matrix(n, m, 4e-4, "bf16", 90 + i).to(DEV) for i, (n, m) in enumerate(shapes)]
    results = []
    for odd in (0, 1):
        W = [w.clone() for w in W0]
        S = [_sketch(n, r, odd if i == 0 else 0, 0, 100 + i)[1] for i, (n, _) in enumerate(shapes)]
        fset = fb.FloraSet(G[1:], W[1:], S[1:]) if odd == 0 else fb.FloraSet(G, W, S)
        seeds = [110 + i for i in range(1 - odd, len(shapes))]
        fset.decompress_apply(seeds, 0.03, 1.0)
        if odd:
            _weights_match(W[0], W0[0], S[0], 110, 0.03)
        want = [oracle_compress(G[i], S[i], 110 + i) for i in range(len(shapes))]
        fset.compress_accumulate(seeds)
        for i in range(1 - odd, len(shapes)):
            assert rel_err(S[i].cpu().numpy(), want[i]) <= TOL["f32"], i
        fset.close()
        results.append(W[1:])
    assert all(torch.equal(x, y) for x, y in zip(*results))


def test_no_memory_for_the_copy_of_the_sketches():
    """A set is made all the same, whichever of its sketches wants the copy (1.6 GB here)."""
    n, m = 1 << 22, 64
    W = [torch.zeros(128, m, dtype=torch.bfloat16, device=DEV), torch.zeros(n, m, dtype=torch.bfloat16, device=DEV)]
    S = [torch.ones(128, 4, device=DEV)[:, :1], torch.ones(n, 1, device=DEV)]
    torch.cuda.empty_cache()
    rest = torch.empty(max(0, torch.cuda.mem_get_info()[0] - (1 << 30)), dtype=torch.uint8, device=DEV)
    try:
        fset = fb.FloraSet(None, W, S)
    finally:
        del rest
        torch.cuda.empty_cache()
    fset.decompress_apply([3, 4], 0.5, 1.0)
    fset.close()
    for i in range(2):
        A = torch.empty(1, m, device=DEV)
        fb.flora_materialize_A(A, 3 + i)
        assert torch.equal(W[i], (-0.5 * A.bfloat16().float()).bfloat16().expand_as(W[i]))


@pytest.mark.parametrize("r,ld", [(61, 64), (30, 32), (7, 8), (101, 104), (253, 256)])
def test_what_lies_behind_a_row_is_not_read(r, ld):
    """Ranks that are no multiple of four, rows 16 bytes apart: TMA reads such a sketch, and what is behind its rows (NaN) stays out of the weights."""
    n, m = 256, 1024
    buf = torch.full((n, ld), float("nan"), device=DEV)
    S = buf[:, :r]
    S.copy_(torch.randn(n, r, generator=torch.Generator().manual_seed(1)))
    W = wl.gaussian_matrix(n, m, 4e-4, "bf16", 6).to(DEV)
    W0 = W.clone()
    fb.flora_decompress_apply(W, S, 14, 0.03, 1.0)
    _weights_match(W, W0, S, 14, 0.03)
    assert buf[:, r:].isnan().all()


@pytest.mark.parametrize("n,m,r", [(2564, 4048, 48), (8200, 1016, 64)])
def test_first_compressions_of_a_shape_inside_a_graph(n, m, r):
    """Matrices a little above the size up to which the general kernels are the quicker: calls that a graph records first need no plan."""
    fb.flora_debug_force_path(0)                                      # (shapes of their own: no plan of another test)
    G, S = wl.gaussian_matrix(n, m, 1e-2, "bf16", 1).to(DEV), torch.zeros(n, r, device=DEV)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        fb.flora_momentum_step(G, S, 0.0, 3)
        fb.flora_compress_accumulate(G, S, 3, r)
    G2 = wl.gaussian_matrix(n, m, 1e-2, "bf16", 4).to(DEV)
    G.copy_(G2)
    graph.replay()
    rows = np.arange(0, n, 257)
    want = 2.0 * oracle_compress(G2[rows].contiguous(), torch.zeros(len(rows), r), 3)
    assert rel_err(S[rows].cpu().numpy(), want) <= TOL["f32"]
    del graph
