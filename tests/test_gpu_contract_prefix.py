"""The contraction of orders m >= 5 by prefixes and pairs (FP32 / BF16 storage, larger
tensors) against the FP64 oracle."""
import numpy as np
import pytest
import torch

import oracle
import synth
from gpu_util import U32, as_f64, contraction_bound

pytestmark = pytest.mark.gpu

tk = pytest.importorskip("paper_2003_10482_gb300")


def prefix_rel(m, n):
    """gamma of the pass's longest chain: a column sum of some 1024 + n prefixes of an
    item and runs of 8 items; a row sum of 8 entries a lane, 5 shuffle levels, runs of
    8 tiles and one rounding of tau; the products of a term 3m + 20.  tau is then
    contracted by the streaming pass, whose own bound is added."""
    return 1.01 * (1024 + n + 8 + 8 + 5 + 8 + 1 + 3 * m + 20) * U32


@pytest.mark.parametrize("m,n,storage,vdt", [(5, 90, "f32", torch.float64), (6, 56, "bf16", torch.float32),
                                             (7, 41, "f32", torch.float64), (8, 33, "f32", torch.float64)])
def test_pass_matches_streaming_pass(m, n, storage, vdt):
    # K[a^{m-2}, a] = K[a^{m-1}] and a . K[a^{m-1}] = K[a^m]: the Hessian-vector
    # product, which the streaming kernel computes, is the reference, within both
    # passes' bounds on the sums of |terms| (the same product of |K| and |a|)
    Kd = tk.tk_build_packed(torch.tensor(synth.small_problem(m, n, 4, salt=1300 + n), device="cuda"), m, storage=storage)
    A = torch.tensor(synth.alpha_like(n, salt=1301), device="cuda").to(vdt)
    G, S = tk.tk_contract(Kd, m, n, A)
    assert tk.tk_status_read(tk.workspace(m, n)) == tk.TK_OK
    G2, S2 = tk.tk_contract(Kd, m, n, A)
    assert torch.equal(G, G2) and torch.equal(S, S2)
    A64 = A.double()
    ref, _ = tk.tk_contract(Kd, m, n, A64, r=m - 2, V=A64)
    mag, _ = tk.tk_contract(Kd.abs(), m, n, A64.abs(), r=m - 2, V=A64.abs())
    ref, mag, a = ref.cpu().numpy(), 1.001 * mag.cpu().numpy(), A64.cpu().numpy()
    tol = prefix_rel(m, n) * mag + contraction_bound(n, mag, "f32", m - 2) + 2 * contraction_bound(n, mag, storage, m, dual=True)
    err = np.abs(G.double().cpu().numpy() - ref)
    assert np.all(err <= tol + (U32 * np.abs(ref) if vdt == torch.float32 else 0.0)), float(np.max(err / tol))
    assert abs(float(S[0]) - a @ ref) <= np.abs(a) @ tol


def test_pass_matches_oracle():
    m, n = 5, 90
    Kd = tk.tk_build_packed(torch.tensor(synth.small_problem(m, n, 4, salt=1390), device="cuda"), m, storage="f32")
    a = synth.alpha_like(n, salt=1391)
    G, S = tk.tk_contract(Kd, m, n, torch.tensor(a, device="cuda"))
    K = as_f64(Kd)
    g_ref, S_ref = oracle.contract(K, a, m)
    g_abs, S_abs = oracle.contract(np.abs(K), np.abs(a), m)
    assert np.all(np.abs(G.cpu().numpy() - g_ref) <= prefix_rel(m, n) * g_abs + contraction_bound(n, g_abs, "f32", m - 2))
    assert abs(float(S[0]) - S_ref) <= prefix_rel(m, n) * S_abs + contraction_bound(n, np.array([S_abs]), "f32", m - 2)[0]
