"""Bit parity of the quantizer's kernels with the oracle at the sizes where each can go wrong: rows that are
not whole 16-byte vectors, a last group of one column, groups of the whole row over several 240-column tiles
with ragged ends, column sums over several tiles on both CTA sizes, more scores than fit in shared memory in
the salient selection, and weights outside the range of the fast division."""
import numpy as np
import pytest

import synth
from oracle import quantize as oq

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qt():
    import paper_2609_00224_gb300 as m
    m.load()
    return m


def same(qt, W, h, group, s, bias, fit_iters=4, rescale_iters=2):
    out = qt.qtea_quantize(torch.from_numpy(W).cuda(), torch.from_numpy(h).cuda(), group_size=group, n_salient=s,
                           bias=bias, fit_iters=fit_iters, rescale_iters=rescale_iters)
    torch.cuda.synchronize()
    ref = oq.quantize(W, h, group, s, bias, fit_iters, rescale_iters)
    for k, v in out.items():
        if s or not k.startswith("residual"):
            got = v.cpu().numpy()
            assert np.array_equal(got.view(ref[k].dtype).reshape(-1), ref[k].reshape(-1)), k


@pytest.mark.parametrize("N,K,group,s,bias", [
    (36, 257, 128, 9, True),       # a last group of one column, 4-byte copies
    (40, 1001, 1001, 13, True),    # one group per row, 4-byte copies, a ragged last tile
    (64, 960, 960, 4, False),      # four whole tiles of 240 columns
    (68, 1204, 1204, 40, True),    # the last tile 4 columns wide
    (500, 384, 128, 12, True),     # column sums over three 240-row tiles, the last ragged
    (260, 5120, 128, 24, False),   # the smaller CTAs of the column sums, three 112-row tiles
    (8, 20000, 128, 300, True),    # more scores than shared memory holds
    (4, 20000, 20000, 20000, False),
])
def test_paths(qt, N, K, group, s, bias):
    W, h = synth.quant_problem(N + 3 * K + s, N, K)
    same(qt, W, h, group, s, bias)


@pytest.mark.parametrize("group", [128, 512])
@pytest.mark.parametrize("scale", [2.0 ** -60, 2.0 ** -110, 2.0 ** 45, 2.0 ** 70])
def test_division_range(qt, group, scale):
    """Some rows far outside the range of the fast division, zeros and an all-zero group among them. (The
    binary16 outputs saturate or vanish there; the codes and v still follow from the float32 values.)"""
    W, h = synth.quant_problem(17, 256, 512)
    W[::5] *= np.float32(scale)
    W[3, :200] = 0.0
    W[:, 7] = 0.0
    W[9, 128:256] = 0.0
    with np.errstate(over="ignore", under="ignore", invalid="ignore"):
        same(qt, W, h, group, 0, True)


def test_fast_division_is_correctly_rounded(qt):
    """One column's sum of one term per round: v = RN(|W| / alpha) for 3,000 groups, with operands whose
    quotients lie close to rounding boundaries (neighbours of products of the divisor)."""
    rng = np.random.default_rng(4)
    K, N = 128, 3000
    W = np.zeros((N, K), np.float32)
    W[:, 0] = rng.uniform(0.5, 2.0, N).astype(np.float32)
    W[:, 1:40] = rng.uniform(0.001, 2.0, (N, 39)).astype(np.float32)
    W[::2, 1] = np.nextafter(W[::2, 0] * np.float32(1.5), np.float32(4))
    same(qt, W, np.ones(K, np.float32), 128, 0, False, fit_iters=3, rescale_iters=3)
