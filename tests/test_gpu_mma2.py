"""GPU parity of the tensor-core kernel on 2-bit codes (2 <= M <= 16, and FP8 residuals at M = 1) against the
fp64 oracle, at the sizes where it can go wrong: the edges of its 256-row tiles and 512-column chunks, groups
that end inside a chunk, batch sizes on both sides of an n8 tile in either form (four rows up to M = 4, eight
beyond), one and two residual steps per chunk and one entry more (which goes to the older low-batch kernel),
scale rows that cannot be copied as vectors, many CTAs on one tile.

Pass rule per element: |y - y_ref| <= 4e-6 * sum_j |x_j * W^[o][j]| + 1e-7. Every operand is exact, a chunk's
products are summed on the tensor core (at most 32 steps, each truncated below 2^-23 of the partial sum: 3.8e-6)
and the rest in fp32, whose errors are an order smaller in practice.
"""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

REL, ABS = 4e-6, 1e-7


@pytest.fixture(scope="module")
def qt():
    import paper_2609_00224_gb300 as m
    m.load()
    return m


def dev(a, dtype=None):
    t = torch.from_numpy(np.ascontiguousarray(a))
    return (t if dtype is None else t.view(dtype)).cuda()


def shifted(t, n):
    """The same values at an address n elements further on."""
    buf = torch.empty(t.numel() + n, dtype=t.dtype, device="cuda")
    buf[n:].copy_(t.reshape(-1))
    return buf[n:].view(t.shape)


def problem(qt, N, K, M, s, group, bias, fp8, seed, shift=0):
    p = synth.make_problem("mma2", N, K, M, s, seed=seed, group_size=group, beta_std=0.002 if bias else 0.0,
                           residual_fp8=fp8)
    lay = qt.qtea_pack_layout(dev(p.T), n_salient=s, group_size=group or K, fmt=qt.QTEA_FMT_2BIT)
    lay.set_options((qt.QTEA_OPT_BIAS if bias else 0) | (qt.QTEA_OPT_RESIDUAL_FP8 if fp8 else 0))
    f16 = lambda a: shifted(dev(np.ascontiguousarray(a).view(np.int16), torch.float16), shift)
    sc = p.alpha.reshape(-1) if not bias else np.stack([p.alpha.reshape(N, -1), p.beta.reshape(N, -1)], axis=-1).reshape(-1)
    return p, dict(x=f16(p.x), layout=lay, row_scale=f16(sc), col_scale=f16(p.v),
                   salient_idx=dev(p.salient_idx) if s else None,
                   residual_vals=(dev(p.residual_vals) if fp8 else f16(p.residual_vals)) if s else None,
                   residual_idx=dev(p.residual_idx) if s else None)


def check(p, y, bias):
    y_ref, bound = oracle.gemv(p.x, p.T, p.alpha, p.v, p.salient_idx, p.residual_vals, p.residual_idx,
                               beta=p.beta if bias else None, group_size=p.group_size or p.K, residual_fp8=p.residual_fp8)
    err, lim = np.abs(y.cpu().numpy().astype(np.float64) - y_ref), REL * bound + ABS
    assert np.all(err <= lim), f"{p.N}x{p.K} M {p.M}: worst normalised error {(err / lim).max():.3g}"


CASES = [  # N, K, M, s, group, bias, fp8
    (4, 128, 2, 4, 0, False, False), (252, 512, 3, 16, 128, True, True), (260, 640, 2, 8, 128, True, False),
    (256, 1024, 4, 64, 128, True, True), (516, 1100, 5, 40, 128, False, True), (1000, 513, 8, 24, 0, True, False),
    (128, 2048, 9, 48, 128, True, True), (300, 127, 12, 0, 0, False, False), (64, 4096, 13, 120, 0, False, True),
    (1028, 3072, 16, 88, 128, True, True), (33, 5, 3, 0, 0, False, False), (16, 14336, 16, 432, 128, False, True),
    (512, 896, 7, 8, 0, True, False), (512, 896, 1, 8, 0, True, True), (4, 28672, 4, 856, 0, False, True), (40, 1536, 6, 96, 128, True, False),
    (256, 512, 4, 32, 0, False, False), (256, 512, 4, 33, 0, False, False), (256, 512, 10, 32, 128, True, True),
    (16, 17408, 2, 520, 0, False, True), (768, 700, 16, 7, 0, True, False),
]


@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("N,K,M,s,group,bias,fp8", CASES)
def test_parity(qt, N, K, M, s, group, bias, fp8, shift):
    p, q = problem(qt, N, K, M, s, group, bias, fp8, seed=N + 3 * K + 5 * M + s, shift=shift)
    assert qt.qtea_gemv_plan([q]) == ["low_batch"]
    y = qt.qtea_gemv(**q)
    y2 = qt.qtea_gemv(**q)
    torch.cuda.synchronize()
    assert qt.qtea_device_status(q["layout"]) == 0
    check(p, y, bias)
    assert torch.equal(y, y2)


@pytest.mark.parametrize("M", [2, 7, 16])
def test_mixed_group_and_graph_replay(qt, M):
    """Problems with and without staged scales in one call, captured in a graph and replayed on other
    activations in the same buffers."""
    specs = [(512, 1024, 32, 128, True, True), (260, 700, 16, 0, False, False), (768, 2048, 0, 128, True, False),
             (1024, 4096, 128, 0, False, True)]
    items = [problem(qt, N, K, M, s, g, b, f, seed=70 + i) for i, (N, K, s, g, b, f) in enumerate(specs)]
    probs = [dict(q, y=torch.empty((M, p.N), dtype=torch.float32, device="cuda")) for p, q in items]
    assert qt.qtea_gemv_plan(probs) == ["low_batch"] * 4
    st, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    st.wait_stream(torch.cuda.current_stream())
    with torch.cuda.graph(graph, stream=st):
        qt.qtea_gemv_grouped(probs)
    for seed in (1, 2):
        for i, (p, _) in enumerate(items):
            p.x[:] = synth.normal_f16(900 + seed, i, p.x.shape, 0.0, 1.0)
            probs[i]["x"].copy_(dev(p.x.view(np.int16), torch.float16))
        graph.replay()
        torch.cuda.synchronize()
        for (p, _), q, spec in zip(items, probs, specs):
            check(p, q["y"], spec[4])


@pytest.mark.parametrize("M", [3, 9])
@pytest.mark.parametrize("value", [30000.0, 2.0 ** -24])
@pytest.mark.parametrize("which", ["alpha", "v"])
def test_extreme_scales(qt, M, value, which):
    """The largest alphas and column scales stay finite, and subnormal ones keep every bit."""
    p, q = problem(qt, 64, 512, M, 0, 128, False, False, seed=8)
    getattr(p, which)[::3] = synth.f16_from_double(value)
    q["row_scale" if which == "alpha" else "col_scale"].copy_(
        dev(np.ascontiguousarray(getattr(p, which)).reshape(-1).view(np.int16), torch.float16))
    check(p, qt.qtea_gemv(**q), False)


@pytest.mark.parametrize("M", [3, 12])
def test_dense_salient_set_graph_replay(qt, M):
    """The older low-batch kernel, captured in a graph and replayed on other activations: as the direct call."""
    items = [problem(qt, N, 2048, M, 512, g, False, False, seed=90 + i) for i, (N, g) in enumerate([(4096, 0), (2048, 128)])]
    probs = [dict(q, y=torch.empty((M, p.N), dtype=torch.float32, device="cuda")) for p, q in items]
    st, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    st.wait_stream(torch.cuda.current_stream())
    with torch.cuda.graph(graph, stream=st):
        qt.qtea_gemv_grouped(probs)
    for _ in range(5):
        for q in probs:
            q["x"].copy_(torch.randn(q["x"].shape, device="cuda").half())
        graph.replay()
        torch.cuda.synchronize()
        y = [q["y"].clone() for q in probs]
        qt.qtea_gemv_grouped(probs)
        torch.cuda.synchronize()
        for a, q in zip(y, probs):
            assert float((a - q["y"]).norm() / q["y"].norm()) < 1e-6
