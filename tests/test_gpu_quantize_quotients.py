"""Single quotients of the quantizer's column sums, one float32 ulp from a change of the stored output: one row, so
that v_j = RN(|W_j| / alpha) is one quotient, and |W_j| = alpha times the midpoint of two binary16 values or a
neighbour of that product, so that a quotient off by an ulp rounds to the other binary16 value in many columns."""
import numpy as np
import pytest

from oracle import quantize as oq

F = np.float32


def quotient_problem(seed, groups=64, group=128):
    """W [1][groups * group] and each group's alpha = sum |W| / 128, which the last column of a group makes exact: the
    others' sum lies between a half and one of 128 alpha, so their difference is a float32 number."""
    rng = np.random.default_rng(seed)
    W, A = np.zeros((groups, group), F), np.zeros(groups, F)
    for g in range(groups):
        a = F(rng.uniform(1.0, 2.0) * 2.0 ** rng.choice([-38, -10, 0, 10, 38]))
        h = rng.uniform(0.55, 1.2, group - 1).astype(np.float16)
        mid = (h.astype(np.float64) + np.nextafter(h, np.float16(4)).astype(np.float64)) / 2  # 12 bits
        w = (mid * np.float64(a)).astype(F)
        step = rng.integers(-1, 2, group - 1)
        w = np.where(step > 0, np.nextafter(w, F(np.inf)), np.where(step < 0, np.nextafter(w, F(0)), w)).astype(F)
        s = F(0)
        for t in w:
            s = F(s + t)
        last = F(F(128) * a - s)
        assert F(s + last) == F(128) * a and last > 0
        W[g] = np.append(w, last) * np.where(rng.random(group) < 0.5, -1, 1)
        A[g] = a
    return W.reshape(1, -1), A


def f16(q):
    return q.astype(np.float16).view(np.uint16)


@pytest.mark.parametrize("seed", [1, 2])
def test_an_ulp_shows(seed):
    """On the CPU: quotients off by one ulp, and those of one multiplication by the rounded reciprocal, change many of the
    outputs, so the GPU test below can fail."""
    W, A = quotient_problem(seed)
    d, a = np.abs(W).reshape(len(A), -1), A[:, None]
    q = d / a
    on = d > a / 2
    for other in (np.nextafter(q, F(np.inf)), np.nextafter(q, F(0)), (d * (F(1) / a)).astype(F)):
        assert (f16(other) != f16(q))[on].mean() > 0.02
    assert on.mean() > 0.9


@pytest.mark.gpu
@pytest.mark.parametrize("seed", [1, 2])
def test_quotients_are_correctly_rounded(seed):
    torch = pytest.importorskip("torch")
    import paper_2609_00224_gb300 as qt
    W, _ = quotient_problem(seed)
    h = np.ones(W.shape[1], F)
    with np.errstate(over="ignore", under="ignore"):
        out = qt.qtea_quantize(torch.from_numpy(W).cuda(), torch.from_numpy(h).cuda(), group_size=128, n_salient=0,
                               bias=False, fit_iters=0, rescale_iters=1)
        ref = oq.quantize(W, h, 128, 0, False, 0, 1)
    torch.cuda.synchronize()
    for k in ("codes", "row_scale", "col_scale"):
        assert np.array_equal(out[k].cpu().numpy().view(ref[k].dtype).reshape(-1), ref[k].reshape(-1)), k
