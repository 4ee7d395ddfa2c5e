"""The build as a product of prefix rows and pair rows: tile edges, panels, ranges
and non-finite features, for FP32 / BF16 storage (tensor cores) and FP64."""
import numpy as np
import pytest
import torch

import oracle
import synth
from gpu_util import U32, U64, UBF16, as_f64

pytestmark = pytest.mark.gpu

tk = pytest.importorskip("paper_2003_10482_gb300")


def rel_bound(d, m, storage):
    """Relative to sum_k prod_j |x|.  FP64: d products of m factors and their sum.
    Otherwise the m feature roundings and m - 3 prefix products; what the
    three-part split leaves out (two residuals of 2^-26, part pairs below 2^-26
    thrice); per chunk of 64 features at most 64 additions in the main
    accumulator and 320 in the one of the smaller part pairs (2^-7 of it), each
    off by an ulp (2u: no rounding mode assumed); two additions per chunk in
    registers."""
    if storage == "f64":
        return 1.01 * (d + m + 2) * U64
    chunks = -(-d // 64)
    k = min(d, 64)
    return 1.01 * (U32 * (m + m) + 5 * 2.0 ** -26 + 2 * U32 * k * (1 + 5 * 2.0 ** -7) + U32 * 2 * chunks)


@pytest.fixture(autouse=True)
def every_size():
    tk.tk_build_set_config(1)
    yield
    tk.tk_build_set_config(0)


@pytest.mark.parametrize("storage", ["f64", "f32", "bf16"])
@pytest.mark.parametrize("m,n,d", [(3, 1, 1), (3, 15, 64), (3, 129, 65), (4, 15, 63), (4, 16, 129), (4, 33, 16), (5, 12, 200),
                                   (7, 6, 17), (4, 45, 1)])
def test_tile_edges(m, n, d, storage):
    X = synth.small_problem(m, n, d, salt=900 + n + d)
    Kh = as_f64(tk.tk_build_packed(torch.tensor(X, device="cuda"), m, storage=storage))
    tol = rel_bound(d, m, storage) * oracle.build(np.abs(X), m)
    if storage == "bf16":
        tol = tol + UBF16 * (np.abs(Kh) + tol)
    assert np.all(np.abs(Kh - oracle.build(X, m)) <= tol + 1e-300)
    assert tk.tk_build_status() == tk.TK_OK


@pytest.mark.parametrize("storage", ["f64", "f32"])
@pytest.mark.parametrize("m,n", [(3, 60), (4, 40), (5, 16)])
def test_ranges_and_panels_give_the_same_bits(m, n, storage):
    X = torch.tensor(synth.small_problem(m, n, 70, salt=950 + n), device="cuda")
    full = tk.tk_build_packed(X, m, storage=storage)
    N = full.numel()
    cuts = [0, 1, N // 7, N // 2, N - 2, N]
    parts = [tk.tk_build_packed(X, m, storage=storage, off_lo=lo, off_hi=hi) for lo, hi in zip(cuts[:-1], cuts[1:])]
    assert torch.equal(torch.cat(parts), full)
    st = torch.cuda.Stream()
    st.wait_stream(torch.cuda.current_stream())
    other = tk.tk_build_packed(X, m, storage=storage, stream=st)  # the library's own memory
    torch.cuda.current_stream().wait_stream(st)
    assert torch.equal(other, full)
    need = tk.lib().tk_build_workspace_size(m, n, 70, tk.dtype_code(storage))
    assert (need == 0) == (storage == "f64")
    for size in (need * 2 // 3, need // 3) if need else ():
        work = torch.empty(size, dtype=torch.uint8, device="cuda")
        K = torch.empty_like(full)
        assert tk.lib().tk_build_packed_work(m, n, 70, X.data_ptr(), 0, 1, tk.dtype_code(storage), 0, N, K.data_ptr(),
                                             work.data_ptr(), size, torch.cuda.current_stream().cuda_stream) == tk.TK_OK
        assert torch.equal(K, full)


@pytest.mark.parametrize("storage", ["f64", "f32"])
def test_non_finite_features_stay_in_their_entries(storage):
    m, n, d = 4, 20, 9
    X = synth.small_problem(m, n, d, salt=960)
    clean = as_f64(tk.tk_build_packed(torch.tensor(X, device="cuda"), m, storage=storage))
    X[3, 2], X[11, 5], X[17, 0] = np.inf, np.nan, 1e30
    K = as_f64(tk.tk_build_packed(torch.tensor(X, device="cuda"), m, storage=storage))
    for off, t in enumerate(oracle.enumerate_tuples(m, n)):
        with np.errstate(all="ignore"):
            x = X[list(t)].astype(np.float64 if storage == "f64" else np.float32)
            terms = x[0] * x[1] * x[2] * x[3]
        if 11 in t:
            assert np.isnan(K[off])
        elif 3 in t and 17 not in t:
            assert np.isinf(terms[2]) and K[off] == terms[2]
        elif 3 not in t and 17 not in t:
            assert K[off] == clean[off]
