"""The single-vector pass over the tensor as a matrix of prefixes x pairs (order 4,
FP32 / BF16 storage, n >= 200): every output against the FP64 oracle."""
import numpy as np
import pytest
import torch

import oracle
import synth
from gpu_util import U32, as_f64

pytestmark = pytest.mark.gpu

tk = pytest.importorskip("paper_2003_10482_gb300")


def pairs_rel(n):
    """gamma of the pass's longest chain: a column sum of at most n prefixes and runs
    of 16 values of b; a row sum of 16 entries a lane, 5 shuffle levels and runs of 8
    tiles; the products of a term (vector conversions, coefficients, weights) 20."""
    return 1.01 * ((n + 16) + 16 + 5 + 8 + 20) * U32


@pytest.mark.parametrize("n,vdt,storage", [(200, torch.float64, "f32"), (211, torch.float32, "bf16")])
def test_pass_matches_oracle(n, vdt, storage):
    m = 4
    Kd = tk.tk_build_packed(torch.tensor(synth.small_problem(m, n, 5, salt=1200 + n), device="cuda"), m, storage=storage)
    A = torch.tensor(synth.alpha_like(n, salt=1201), device="cuda").to(vdt)
    V = torch.tensor(synth.alpha_like(n, salt=1202), device="cuda").to(vdt)
    G, S = tk.tk_contract(Kd, m, n, A)
    HV, _ = tk.tk_contract(Kd, m, n, A, r=2, V=V)
    K, a, v = as_f64(Kd), A.double().cpu().numpy(), V.double().cpu().numpy()
    g_ref, S_ref = oracle.contract(K, a, m)
    h_ref = oracle.hvp(K, a, v, m)
    g_abs, S_abs = oracle.contract(np.abs(K), np.abs(a), m)
    h_abs = oracle.hvp(np.abs(K), np.abs(a), np.abs(v), m)
    out = U32 if vdt == torch.float32 else 0.0  # results rounded to the vector type
    assert np.all(np.abs(G.double().cpu().numpy() - g_ref) <= pairs_rel(n) * g_abs + out * np.abs(g_ref))
    assert abs(float(S[0]) - S_ref) <= pairs_rel(n) * S_abs
    # the product rule doubles the rounded terms of a product
    assert np.all(np.abs(HV.double().cpu().numpy() - h_ref) <= 2 * pairs_rel(n) * h_abs + out * np.abs(h_ref))
    if vdt == torch.float64:
        y = torch.tensor(synth.alpha_like(n, salt=1203), device="cuda")
        F, grad, gn = tk.tk_objective(Kd, m, n, A, y, 0.7)
        assert torch.allclose(grad, G + 0.7 * A - y, rtol=1e-13, atol=1e-13 * float(grad.abs().max()))
        assert float(F[0]) == pytest.approx(float(S[0] / m + 0.35 * (A @ A) - y @ A), rel=1e-13, abs=1e-12)
        assert float(gn[0]) == pytest.approx(float(grad.norm()), rel=1e-13)


def test_pass_is_reproducible_and_leaves_other_plans_alone():
    m, n = 4, 203
    Kd = tk.tk_build_packed(torch.tensor(synth.small_problem(m, n, 4, salt=1210), device="cuda"), m, storage="f32")
    K5 = tk.tk_build_packed(torch.tensor(synth.small_problem(5, 20, 3, salt=1211), device="cuda"), 5, storage="f32")
    A = torch.tensor(synth.alpha_like(n, salt=1212), device="cuda")
    work = tk.new_workspace(int(tk.lib().tk_contract_workspace_size(m, n, 1)), A.device)
    G, S = tk.tk_contract(Kd, m, n, A, work=work)
    G5, _ = tk.tk_contract(K5, 5, 20, A[:20].clone(), work=work)
    HV, _ = tk.tk_contract(Kd, m, n, A, r=2, V=A, work=work)
    G5b, _ = tk.tk_contract(K5, 5, 20, A[:20].clone(), work=work)
    G2, S2 = tk.tk_contract(Kd, m, n, A, work=work)
    assert torch.equal(G, G2) and torch.equal(S, S2) and torch.equal(G5, G5b)
    assert torch.allclose(HV, G, rtol=0, atol=1e-5 * float(G.abs().max()))
    # a workspace of the streaming pass's size still serves (the streaming pass)
    small = tk.new_workspace(8 << 20, A.device)
    G3, S3 = tk.tk_contract(Kd, m, n, A, work=small)
    assert torch.allclose(G3, G, rtol=0, atol=1e-5 * float(G.abs().max()))
