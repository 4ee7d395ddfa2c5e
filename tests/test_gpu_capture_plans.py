"""Passes that keep no plan in the workspace, recorded into a CUDA graph: the replay
gives the direct call's result; replayed after another pass has planned the
workspace it writes nothing, reports that, and leaves the other's plan usable."""
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu

tk = pytest.importorskip("paper_2003_10482_gb300")


def capture(fn):
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        out = fn()
    return g, out


def build(m, n):
    return tk.tk_build_packed(torch.tensor(synth.small_problem(m, n, 4, salt=1300 + n), device="cuda"), m, storage="f32")


@pytest.mark.parametrize("name,m,n", [("pairs", 4, 201), ("prefix", 6, 57), ("hessian", 4, 41)])
def test_replay_over_another_plan_does_nothing(name, m, n):
    K, K2 = build(m, n), build(3, 45)
    a = torch.tensor(synth.alpha_like(n, salt=1301), device="cuda")
    A2 = torch.tensor(synth.alpha_like(8 * 45, salt=1302), device="cuda").reshape(8, 45).contiguous()
    work = tk.new_workspace(256 << 20, a.device)
    out_buf = torch.empty((n, n) if name == "hessian" else n, dtype=torch.float64, device=a.device)

    def call():
        if name == "hessian":
            rc = tk.lib().tk_hessian(m, n, tk.TK_F32, K.data_ptr(), a.data_ptr(), out_buf.data_ptr(), work.data_ptr(),
                                     work.numel(), torch.cuda.current_stream().cuda_stream)
            assert rc == tk.TK_OK
        else:
            tk.tk_contract(K, m, n, a, G=out_buf.view(1, n), work=work)
        return out_buf

    ref = call().clone()
    graph, out = capture(call)
    graph.replay()
    torch.cuda.synchronize()
    assert torch.allclose(out, ref, rtol=0, atol=1e-12 * float(ref.abs().max()))
    # the tensor-core / rows pass plans the workspace, the replay must not touch it
    want = tk.tk_contract(K2, 3, 45, A2, work=work)[0].clone()
    out.fill_(7.0)
    graph.replay()
    torch.cuda.synchronize()
    assert tk.tk_status_read(work) == tk.TK_EINVAL
    assert bool((out == 7.0).all())
    again = tk.tk_contract(K2, 3, 45, A2, work=work)[0]
    assert tk.tk_status_read(work) == tk.TK_OK
    assert torch.equal(want, again)


def test_batched_rows_first_call_under_capture():
    """Without its plan the rows pass leaves a captured call to the other passes."""
    m, n, B = 4, 48, 6
    K = build(m, n)
    A = torch.tensor(synth.alpha_like(B * n, salt=1303), device="cuda").reshape(B, n).contiguous()
    rows, S = tk.tk_contract(K, m, n, A)
    work = tk.new_workspace(64 << 20, A.device)
    one, _ = tk.tk_contract(K, m, n, A[0], work=work)
    graph, (G, _) = capture(lambda: tk.tk_contract(K, m, n, A, work=work))
    graph.replay()
    torch.cuda.synchronize()
    assert tk.tk_status_read(work) == tk.TK_OK
    assert torch.equal(G[0], one.reshape(-1))  # the single-vector pass
    assert torch.allclose(G, rows, rtol=0, atol=1e-5 * float(rows.abs().max()))


def test_solves_of_changing_sizes_share_a_workspace():
    """A solve's Hessian region moves with its sizes, over what an earlier solve kept there."""
    K = {n: build(4, n) for n in (30, 64, 130)}
    y = {n: torch.tensor(synth.alpha_like(n, salt=1304), device="cuda") for n in K}

    def solve(n, B):
        lam = torch.linspace(0.8, 1.2, B, dtype=torch.float64, device="cuda")
        return tk.tk_solve_dual(K[n], 4, n, y[n], lam, method="newton_full", tol=0.0, rel_gap=1e-9, max_iter=30)[0]

    tk._solve_ws.clear()
    order = [(130, 8), (64, 1), (30, 8), (130, 1), (64, 8), (64, 2), (30, 2), (130, 4), (64, 4)]
    first = {c: solve(*c).clone() for c in order}
    for c in order[::-1] + order:
        again = solve(*c)
        # the FP64 sums of the Hessian pass may differ in the last bits
        assert torch.allclose(again, first[c], rtol=0, atol=1e-6 * float(first[c].abs().max())), c
