"""Activations of a wide range on the tensor-core kernel with staged B operands, against the fp64 oracle: one massive
value per 512-column chunk beside activations down to 2^-36 of it, with codes 0 at the massive columns in part of
the rows, where an error relative to the massive value shows. v*x is held as an fp16 pair, exact down to 2^-28 of
the chunk's largest and within 2^-50 of it below; products 2^24 times the chunk's mean are taken out and added in fp32,
as infinities and NaN are. (2-bit codes at M >= 5 take 2T v in A instead, exact below |v| = 2^15; with larger v the sum
is formed in fp32.)

Pass rule per element: |y - y_ref| <= 2e-6 * sum_j |x_j * W^[o][j]|, nothing absolute. The pairs' errors stay below 2^-26
of a chunk's mean product; the tensor core truncates each of a chunk's at most 35 steps below 2^-24 of the partial
sum, which over terms of either sign stays a small part of the bound: 2e-6 is 34 roundings of the whole bound.
"""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

REL = 2e-6


@pytest.fixture(scope="module")
def qt():
    import paper_2609_00224_gb300 as m
    m.load()
    return m


def dev(a, dtype=None):
    t = torch.from_numpy(np.ascontiguousarray(a))
    return (t if dtype is None else t.view(dtype)).cuda()


def operands(qt, p, fmt, bias, fp8):
    lay = qt.qtea_pack_layout(dev(p.T), n_salient=p.s, group_size=p.group_size or p.K,
                              fmt=qt.QTEA_FMT_BASE3 if fmt == "base3" else qt.QTEA_FMT_2BIT)
    lay.set_options((qt.QTEA_OPT_BIAS if bias else 0) | (qt.QTEA_OPT_RESIDUAL_FP8 if fp8 else 0))
    f16 = lambda a: dev(np.ascontiguousarray(a).view(np.int16), torch.float16)
    sc = p.alpha.reshape(-1) if not bias else np.stack([p.alpha.reshape(p.N, -1), p.beta.reshape(p.N, -1)], axis=-1).reshape(-1)
    return dict(x=f16(p.x), layout=lay, row_scale=f16(sc), col_scale=f16(p.v),
                salient_idx=dev(p.salient_idx) if p.s else None,
                residual_vals=(dev(p.residual_vals) if fp8 else f16(p.residual_vals)) if p.s else None,
                residual_idx=dev(p.residual_idx) if p.s else None)


FORMS = [("base3", 1), ("base3", 3), ("base3", 6), ("base3", 16), ("2bit", 1), ("2bit", 2), ("2bit", 4), ("2bit", 7),
         ("2bit", 16)]


def call(qt, p, fmt, bias, fp8):
    q = operands(qt, p, fmt, bias, fp8)
    assert qt.qtea_gemv_plan([q]) == ["base3_mma" if fmt == "base3" else "low_batch"]
    y = qt.qtea_gemv(**q)
    torch.cuda.synchronize()
    assert qt.qtea_device_status(q["layout"]) == 0
    return y.cpu().numpy().astype(np.float64)


@pytest.mark.parametrize("fmt,M", FORMS)
@pytest.mark.parametrize("std", [0.1, 1e-3, 2.0 ** -21])
@pytest.mark.parametrize("K,group", [(1100, 128), (2048, 0)])
def test_massive_beside_small(qt, fmt, M, std, K, group):
    N, s, fp8 = 260, 24, fmt == "2bit" and M == 1  # 2-bit at M = 1: this kernel takes the FP8 residual
    p = synth.make_problem("range", N, K, M, s, seed=K + M, group_size=group, residual_fp8=fp8, x_std=std)
    hi = [6e4, 3e4, 5e4, 2e4, 6e4]
    for ch in range((K + 511) // 512):  # one per chunk, its codes 0 in every second row; no residual there
        c = int(synth.plant_massive(p.x, 10 * ch + M, [hi[ch]], lo=512 * ch, hi=512 * ch + 64)[0])
        p.T[::2, c] = 0
        p.salient_idx[p.salient_idx == c] = c + 1
    p.salient_idx[:] = np.unique(np.concatenate([p.salient_idx, np.arange(K - 40, K)]))[:s]
    y_ref, bound = oracle.gemv(p.x, p.T, p.alpha, p.v, p.salient_idx, p.residual_vals, p.residual_idx,
                               group_size=p.group_size or K, residual_fp8=fp8)
    err = np.abs(call(qt, p, fmt, False, fp8) - y_ref)
    assert np.all(err <= REL * bound), f"worst {(err / bound).max():.3g} of the bound"


@pytest.mark.parametrize("fmt,M", FORMS)
def test_spread_over_every_binade(qt, fmt, M):
    """Magnitudes of x from 2^-24 to 2^15 in every chunk, of v from 2^-14 to 1."""
    N, K, fp8 = 64, 1536, fmt == "2bit" and M == 1
    p = synth.make_problem("spread", N, K, M, 16, seed=M, residual_fp8=fp8)
    rng = np.random.default_rng(M)
    sign = rng.choice([-1.0, 1.0], (M, K))
    p.x[:] = (sign * 2.0 ** rng.uniform(-24, 15, (M, K))).astype(np.float16).view(np.uint16)
    p.v[:] = (2.0 ** rng.uniform(-14, 0, K)).astype(np.float16).view(np.uint16)
    y_ref, bound = oracle.gemv(p.x, p.T, p.alpha, p.v, p.salient_idx, p.residual_vals, p.residual_idx, residual_fp8=fp8)
    err = np.abs(call(qt, p, fmt, False, fp8) - y_ref)
    assert np.all(err <= REL * bound), f"worst {(err / bound).max():.3g} of the bound"


@pytest.mark.parametrize("fmt,M", FORMS)
@pytest.mark.parametrize("group,bias", [(0, False), (128, False)])
def test_infinities_and_nan_reach_their_rows_only(qt, fmt, M, group, bias):
    """A column whose activation is infinite or NaN counts in the rows with a non-zero code (or a residual value)
    there and in no other."""
    N, K, s, fp8 = 132, 1100, 40, fmt == "2bit" and M == 1
    p = synth.make_problem("inf", N, K, M, s, seed=7 + M, group_size=group, residual_fp8=fp8)
    sal = int(p.salient_idx[21])
    bad = {3: np.inf, 700: -np.inf, 1099: np.nan, sal: np.inf}
    x = p.x.view(np.float16)
    finite = x.astype(np.float64).copy()
    for i, (c, value) in enumerate(bad.items()):
        m = (i * 3) % M
        x[m, c] = value
        finite[m, c] = 0.0
        p.T[::3, c] = 0
    y_ref, bound = oracle.gemv(finite.astype(np.float16).view(np.uint16), p.T, p.alpha, p.v, p.salient_idx, p.residual_vals,
                               p.residual_idx, group_size=group or K, residual_fp8=fp8)
    pos = synth.residual_positions(p.residual_idx, s)
    special = np.zeros((M, N))
    with np.errstate(invalid="ignore"):
        for i, (c, value) in enumerate(bad.items()):
            m = (i * 3) % M
            special[m] += np.where(p.T[:, c] != 0, np.sign(p.T[:, c] + 0.5) * value, 0.0)
            for k in np.flatnonzero(p.salient_idx == c):
                rv = oracle_value(p, k, fp8)
                rows = 4 * np.arange(N // 4) + pos[:, k]
                special[m, rows] += np.where(rv != 0, np.sign(rv) * value, np.nan)
        y = call(qt, p, fmt, bias, fp8)
    ok = special == 0
    assert np.array_equal(y[~ok], special[~ok], equal_nan=True)
    assert np.all(np.abs(y - y_ref)[ok] <= REL * bound[ok])
    assert ok.sum() > M * N / 8 and (~ok).sum() > 0


@pytest.mark.parametrize("fmt,M", FORMS + [("2bit", 5), ("2bit", 9)])
@pytest.mark.parametrize("group,bias", [(0, False), (0, True), (128, True)])
def test_column_scales_of_any_size(qt, fmt, M, group, bias):
    """|v| from fp16's smallest to its largest (2 v is no fp16 number from 2^15 on)."""
    N, K, fp8 = 132, 1100, fmt == "2bit" and M == 1
    p = synth.make_problem("v", N, K, M, 24, seed=11 + M, group_size=group, beta_std=0.002 if bias else 0.0, residual_fp8=fp8)
    v = p.v.view(np.float16)
    v[5::97] = 65504.0
    v[6::97] = -32768.0
    v[7::97] = 32752.0
    v[8::97] = 2.0 ** -24
    y_ref, bound = oracle.gemv(p.x, p.T, p.alpha, p.v, p.salient_idx, p.residual_vals, p.residual_idx,
                               beta=p.beta if bias else None, group_size=group or K, residual_fp8=fp8)
    err = np.abs(call(qt, p, fmt, bias, fp8) - y_ref)
    assert np.all(err <= REL * bound), f"worst {(err / bound).max():.3g} of the bound"


def oracle_value(p, k, fp8):
    """The residual values of salient entry k as float64."""
    r = p.residual_vals[:, k]
    if not fp8:
        return r.view(np.float16).astype(np.float64)
    return torch.from_numpy(np.ascontiguousarray(r)).view(torch.float8_e4m3fn).double().numpy()


@pytest.mark.parametrize("fmt,M", [("base3", 2), ("base3", 5), ("base3", 16), ("2bit", 3), ("2bit", 12)])
@pytest.mark.parametrize("massive", [False, True])
def test_row_scales_far_apart(qt, fmt, M, massive):
    """|alpha| of 30000, 1e-4, 2^-24 and 0 in neighbouring rows and groups: the small ones keep every bit, also where
    activations of 2^-21 stand beside one of 6e4."""
    N, K = 132, 700
    p = synth.make_problem("alpha", N, K, M, 0, seed=21 + M, group_size=128, x_std=2.0 ** -21 if massive else 1.0)
    if massive:
        synth.plant_massive(p.x, M, [6e4], lo=0, hi=100)
        synth.plant_massive(p.x, M, [6e4], lo=600, hi=700)
    alpha = p.alpha.view(np.float16)
    alpha[1::5] = 1e-4
    alpha[2::5] = 2.0 ** -24
    alpha[3::5] = 30000.0
    alpha[3::10, 1] = 1.2e-4
    alpha[4::10] = 0.0
    y_ref, bound = oracle.gemv(p.x, p.T, p.alpha, p.v, p.salient_idx, p.residual_vals, p.residual_idx, group_size=128)
    err = np.abs(call(qt, p, fmt, False, False) - y_ref)
    assert np.all(err <= REL * bound), f"worst {np.nanmax(err / np.maximum(bound, 1e-30)):.3g} of the bound"


@pytest.mark.parametrize("M", [5, 9, 16])
@pytest.mark.parametrize("K,group,bias", [(256, 128, True), (370, 128, True), (768, 128, False), (700, 0, True)])
def test_small_errors_where_sums_were_fp32(qt, M, K, group, bias):
    """2-bit calls at M >= 5 with a scale map of no whole 16-byte vectors, or one beta per row: products of 11 bits
    (v*x split), not of 22, whose truncated sums leave 1.1e-7 of the outputs' norm; fp32 sums leave 0.75e-7 to 0.9e-7."""
    p = synth.make_problem("small", 2048, K, M, 0, seed=K + M, group_size=group, beta_std=0.002 if bias else 0.0)
    y_ref, _ = oracle.gemv(p.x, p.T, p.alpha, p.v, p.salient_idx, p.residual_vals, p.residual_idx,
                           beta=p.beta if bias else None, group_size=group or K)
    y = call(qt, p, "2bit", bias, False)
    assert np.linalg.norm(y - y_ref) <= 0.8e-7 * np.linalg.norm(y_ref)
