"""The Hessian pass of orders 3 and 4 at the edges of its 8 x 32 tiles, its blocks of
i and its runs of b, element by element against the oracle's dense Hessian."""
import numpy as np
import pytest
import torch

import oracle
import synth
from gpu_util import as_f64, hessian_bound, round_storage

pytestmark = pytest.mark.gpu

tk = pytest.importorskip("paper_2003_10482_gb300")


@pytest.mark.parametrize("storage", ["f64", "f32", "bf16"])
@pytest.mark.parametrize("m,n", [(3, 1), (3, 8), (3, 33), (3, 72), (4, 2), (4, 7), (4, 8), (4, 9), (4, 31), (4, 32), (4, 41), (4, 65)])
def test_tile_edges(m, n, storage):
    # chain of roundings: a run of b (at most 64), a block of i, 8 rows, 5 shuffle
    # levels and the products, below hessian_bound's max(., 64) + 5 + 12 + 3m + 8
    X = synth.small_problem(m, n, 3, salt=1000 + n)
    Kt = round_storage(oracle.build(X, m), storage)
    a = synth.alpha_like(n, salt=1001 + n)
    H = tk.tk_hessian(Kt.cuda(), m, n, torch.tensor(a, device="cuda")).cpu().numpy()
    Kr = as_f64(Kt)
    tol = hessian_bound(n, m, oracle.hessian(np.abs(Kr), np.abs(a), m), storage)
    assert np.all(np.abs(H - oracle.hessian(Kr, a, m)) <= tol)
    assert np.array_equal(H, H.T)


def test_passes_share_a_workspace_with_other_orders():
    # the sums of orders 3 and 4 overwrite a plan of another order in the same workspace
    n = 20
    a = torch.tensor(synth.alpha_like(n, salt=1010), device="cuda")
    want = {}
    for m in (4, 5, 3, 5, 4):
        K = tk.tk_build_packed(torch.tensor(synth.small_problem(m, n, 3, salt=1011), device="cuda"), m, storage="f64")
        H = tk.tk_hessian(K, m, n, a)
        G, _ = tk.tk_contract(K, m, n, a)
        assert torch.allclose(H @ a, G, rtol=1e-11, atol=1e-11 * float(G.abs().max()))
        assert torch.allclose(want.setdefault(m, H), H, rtol=1e-13, atol=1e-13 * float(H.abs().max()))
