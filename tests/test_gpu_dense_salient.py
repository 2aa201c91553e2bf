"""GPU parity of the kernels that serve layouts whose salient set is too dense for the tensor-core kernel with staged B
operands (more than 32 entries per 512 columns), against the fp64 oracle: the table lookup (base-3 codes, M = 1, with and
without scale groups), the fixed-point kernel (base-3, 2 <= M <= 4), the general kernel for the paper's storage
(base-3, M >= 5) and the older low-batch and general kernels (2-bit codes, M >= 2), single and grouped, on ordinary
and on massive activations.

Pass rule per element: |y - y_ref| <= 1e-4 * sum_j |x_j * W^[o][j]| + 1e-6, the rule of these kernels' other tests.
"""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

REL, ABS = 1e-4, 1e-6
STORAGE = [(0, False, False), (128, False, False), (128, True, False), (128, True, True), (0, False, True)]


@pytest.fixture(scope="module")
def qt():
    import paper_2609_00224_gb300 as m
    m.load()
    return m


def dev(a, dtype=None):
    t = torch.from_numpy(np.ascontiguousarray(a))
    return (t if dtype is None else t.view(dtype)).cuda()


def problem(qt, fmt, N, K, M, s, group, bias, fp8, seed, massive=()):
    p = synth.make_problem("dense", N, K, M, s, seed=seed, group_size=group, beta_std=0.002 if bias else 0.0,
                           residual_fp8=fp8)
    if massive:
        synth.plant_massive(p.x, seed, massive)
    lay = qt.qtea_pack_layout(dev(p.T), n_salient=s, group_size=group or K,
                              fmt=qt.QTEA_FMT_BASE3 if fmt == "base3" else qt.QTEA_FMT_2BIT)
    lay.set_options((qt.QTEA_OPT_BIAS if bias else 0) | (qt.QTEA_OPT_RESIDUAL_FP8 if fp8 else 0))
    f16 = lambda a: dev(np.ascontiguousarray(a).view(np.int16), torch.float16)
    sc = p.alpha.reshape(-1) if not bias else np.stack([p.alpha.reshape(N, -1), p.beta.reshape(N, -1)], axis=-1).reshape(-1)
    return p, dict(x=f16(p.x), layout=lay, row_scale=f16(sc), col_scale=f16(p.v), salient_idx=dev(p.salient_idx),
                   residual_vals=dev(p.residual_vals) if fp8 else f16(p.residual_vals),
                   residual_idx=dev(p.residual_idx))


def check(p, y):
    y_ref, bound = oracle.gemv(p.x, p.T, p.alpha, p.v, p.salient_idx, p.residual_vals, p.residual_idx, beta=p.beta,
                               group_size=p.group_size or p.K, residual_fp8=p.residual_fp8)
    err, lim = np.abs(y.cpu().numpy().astype(np.float64) - y_ref), REL * bound + ABS
    assert np.all(err <= lim), f"{p.N}x{p.K} M {p.M}: worst normalised error {(err / lim).max():.3g}"


def base3_kernel(M):
    return "lut" if M == 1 else "base3_fixed" if M <= 4 else "paper"


@pytest.mark.parametrize("M", [1, 2, 4, 6, 16])
@pytest.mark.parametrize("group,bias,fp8", STORAGE)
@pytest.mark.parametrize("N,K,s", [(260, 1024, 80), (132, 1100, 512), (1028, 2048, 200)])
def test_base3(qt, M, group, bias, fp8, N, K, s):
    p, q = problem(qt, "base3", N, K, M, s, group, bias, fp8, seed=N + K + 7 * M)
    assert qt.qtea_gemv_plan([q]) == [base3_kernel(M)]
    y = qt.qtea_gemv(**q)
    torch.cuda.synchronize()
    assert qt.qtea_device_status(q["layout"]) == 0
    check(p, y)


@pytest.mark.parametrize("M", [1, 3, 8])
def test_base3_massive_activations(qt, M):
    p, q = problem(qt, "base3", 512, 4096, M, 400, 128, True, True, seed=31 + M, massive=(8000.0, 3000.0, 500.0))
    assert qt.qtea_gemv_plan([q]) == [base3_kernel(M)]
    check(p, qt.qtea_gemv(**q))


@pytest.mark.parametrize("M", [2, 4, 5, 8, 16])
@pytest.mark.parametrize("group,bias,fp8", STORAGE)
@pytest.mark.parametrize("N,K,s", [(260, 1024, 80), (132, 1100, 512), (1028, 2048, 200)])
def test_2bit(qt, M, group, bias, fp8, N, K, s):
    p, q = problem(qt, "2bit", N, K, M, s, group, bias, fp8, seed=N + K + 7 * M)
    assert qt.qtea_gemv_plan([q])[0] in ("low_batch", "paper", "generic")
    y = qt.qtea_gemv(**q)
    torch.cuda.synchronize()
    assert qt.qtea_device_status(q["layout"]) == 0
    check(p, y)


@pytest.mark.parametrize("fmt", ["base3", "2bit"])
@pytest.mark.parametrize("M", [1, 3, 6])
def test_grouped_with_sparse_ones(qt, fmt, M):
    """Dense and sparse salient sets in one call: each problem by its own kernel."""
    specs = [(512, 1024, 100, 128, True, True), (260, 700, 16, 0, False, False), (256, 2048, 600, 128, True, False),
             (768, 1024, 96, 0, False, False)]
    items = [problem(qt, fmt, N, K, M, s, g, b, f, seed=50 + i) for i, (N, K, s, g, b, f) in enumerate(specs)]
    plan = qt.qtea_gemv_plan([q for _, q in items])
    if fmt == "base3":
        assert plan == [base3_kernel(M), "base3_mma", base3_kernel(M), base3_kernel(M)]
    for (p, _), y in zip(items, qt.qtea_gemv_grouped([q for _, q in items])):
        check(p, y)


@pytest.mark.parametrize("fmt", ["base3", "2bit"])
@pytest.mark.parametrize("M", [1, 2, 4, 5, 16])
@pytest.mark.parametrize("s", [8, 64])
@pytest.mark.parametrize("fp8", [False, True])
@pytest.mark.parametrize("bias", [False, True])
def test_one_group_of_128_columns(qt, fmt, M, s, fp8, bias):
    """K = 128: groups of 128 columns are one group per row, and the scales pairs with beta."""
    p, q = problem(qt, fmt, 260, 128, M, s, 128, bias, fp8, seed=3 * M + s)
    y = qt.qtea_gemv(**q)
    torch.cuda.synchronize()
    check(p, y)
