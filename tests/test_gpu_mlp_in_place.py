"""GPU: the tuner network's outputs in the memory of its inputs (their start, or a piece that begins inside them)."""
import ctypes

import pytest

torch = pytest.importorskip("torch")

from oracle import mlp as omlp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B", [1, 16, 17, 100, 2000, 24001])
@pytest.mark.parametrize("offset", [0, 36])
def test_outputs_over_inputs(B, offset):
    import paper_2204_06666_gb300 as eh
    g = torch.Generator().manual_seed(B)
    X = torch.randn(B * 16 + 64, generator=g).cuda()
    P = torch.from_numpy(omlp.init(7)).float().cuda()
    ws = torch.empty(int(eh._lib.ehyb_mlp_workspace_bytes(B)), dtype=torch.uint8, device="cuda")
    ref = torch.empty(B * 4, device="cuda")
    s = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    for x, out in ((X, ref), (X, X[offset:])):
        assert eh._lib.ehyb_mlp_forward(P.data_ptr(), x.data_ptr(), B, out.data_ptr(), ws.data_ptr(), s) == 0
    assert torch.equal(X[offset:offset + B * 4], ref)
