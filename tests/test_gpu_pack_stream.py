"""A layout packed on a non-blocking stream while the default stream is busy is ready for that stream: its
workspaces (partial rows of split tiles, counters: zero reads as "not written yet") are zeroed in the order of
the packing stream, not behind the default stream's work. The device memory they come from is filled with
other values first, and each problem splits its tiles over several CTAs.

Pass rule per element: |y - y_ref| <= 1e-4 * sum_j |x_j * W^[o][j]| + 1e-6, the rule of the path with the
coarsest activations (16-bit fixed point).
"""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

BUSY_CYCLES = 400_000_000  # of torch.cuda._sleep on the default stream: about 0.2 s


@pytest.fixture(scope="module")
def qt():
    import paper_2609_00224_gb300 as m
    m.load()
    return m


def dev(a, dtype=None):
    t = torch.from_numpy(np.ascontiguousarray(a))
    return (t if dtype is None else t.view(dtype)).cuda()


@pytest.mark.parametrize("fmt,M,s", [
    ("base3", 1, 32), ("base3", 3, 32), ("base3", 16, 32),  # tensor-core kernel
    ("base3", 1, 1600),                                     # table lookup (dense salient set)
    ("2bit", 1, 32), ("2bit", 4, 32), ("2bit", 16, 32),     # stream-K, tensor-core kernel
    ("2bit", 4, 1600),                                      # the older low-batch kernel
])
def test_pack_on_side_stream(qt, fmt, M, s):
    N, K = 512, 16384
    p = synth.make_problem("pack_stream", N, K, M, s, seed=3 * M + s)
    f16 = lambda a: dev(np.ascontiguousarray(a).view(np.int16), torch.float16)
    codes = dev(p.T)
    args = dict(x=f16(p.x), row_scale=f16(p.alpha.reshape(-1)), col_scale=f16(p.v), salient_idx=dev(p.salient_idx),
                residual_vals=f16(p.residual_vals), residual_idx=dev(p.residual_idx))
    y = torch.zeros((M, N), dtype=torch.float32, device="cuda")

    def pack_and_call():
        lay = qt.qtea_pack_layout(codes, n_salient=s, fmt=qt.QTEA_FMT_BASE3 if fmt == "base3" else qt.QTEA_FMT_2BIT)
        if fmt == "2bit" and M == 1:
            lay.set_options(qt.QTEA_OPT_STREAM_K)
        qt.qtea_gemv(layout=lay, y=y, **args)
        return lay

    pack_and_call()  # loads the kernels: the first launch of one waits for the device
    y.zero_()
    # blocks of the workspaces' sizes, freed holding 1.0s: the next allocations find them
    dirty = [torch.ones(n, dtype=torch.float32, device="cuda") for n in (1 << 14, 1 << 18, 1 << 19, 1 << 20, 1 << 21)]
    torch.cuda.synchronize()
    del dirty
    torch.cuda.empty_cache()
    side = torch.cuda.Stream()
    torch.cuda._sleep(BUSY_CYCLES)
    with torch.cuda.stream(side):
        lay = pack_and_call()
        side.synchronize()
    busy = not torch.cuda.default_stream().query()
    torch.cuda.synchronize()
    assert qt.qtea_device_status(lay) == 0
    assert busy, "the default stream was idle before the call ended: nothing was tested"
    y_ref, bound = oracle.gemv(p.x, p.T, p.alpha, p.v, p.salient_idx, p.residual_vals, p.residual_idx)
    err = np.abs(y.cpu().numpy().astype(np.float64) - y_ref)
    assert np.all(err <= 1e-4 * bound + 1e-6)
