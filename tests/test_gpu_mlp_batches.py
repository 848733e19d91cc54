"""GPU: the fused tuner-network step at the batch sizes where its split can go wrong (less than one block's 16
samples, one block, a last block with one sample, more samples than blocks), against the FP64 oracle, with the
workspace exactly as large as the library asks for."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import mlp as omlp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B", [1, 13, 15, 16, 17, 31, 33, 150, 2000, 4001, 24001])
def test_step_at_batch_edges(B):
    import paper_2204_06666_gb300 as eh
    rng = np.random.default_rng(B)
    X, T = rng.standard_normal((B, 16)).astype(np.float32), rng.standard_normal((B, 4)).astype(np.float32)
    th = (omlp.init(7) + rng.uniform(-0.05, 0.05, omlp.NPARAM)).astype(np.float32)
    Xd, Td, P = (torch.from_numpy(a).cuda() for a in (X, T, th))
    need = int(eh._lib.ehyb_mlp_workspace_bytes(B))
    assert need == B * 396 * 4
    guard = 4096
    ws = torch.full((need // 4 + guard,), 777.0, device="cuda")
    g, L = torch.full_like(P, np.nan), torch.full((1,), np.nan, device="cuda")
    s = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    st = eh._lib.ehyb_mlp_loss_grad(P.data_ptr(), Xd.data_ptr(), Td.data_ptr(), B, g.data_ptr(), L.data_ptr(),
                                    ws.data_ptr(), s)
    out = torch.full((B, 4), np.nan, device="cuda")
    st2 = eh._lib.ehyb_mlp_forward(P.data_ptr(), Xd.data_ptr(), B, out.data_ptr(), ws.data_ptr(), s)
    torch.cuda.synchronize()
    assert st == 0 and st2 == 0
    assert bool((ws[need // 4:] == 777.0).all())         # nothing written past the workspace
    Lo, go = omlp.grad(th.astype(np.float64), X.astype(np.float64), T.astype(np.float64))
    oo, _ = omlp.forward(th.astype(np.float64), X.astype(np.float64))
    # FP32 chains of at most 16 + 64 + 64 (forward), 4 + 64 (backward) and 24001/1216 + 152 (batch) terms: about
    # 400 roundings of 2^-24 on terms of one size, 2.4e-5 of their norm; the oracle test's bars are wider
    assert abs(L.item() - Lo) <= 1e-5 * abs(Lo)
    gd = g.cpu().numpy().astype(np.float64)
    assert np.linalg.norm(gd - go) <= 1e-4 * np.linalg.norm(go)
    assert np.allclose(out.cpu().numpy(), oo, rtol=1e-4, atol=1e-5)
