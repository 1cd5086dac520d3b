"""bench.py's list of the kernels that a call launches, read from the captured call, on the
routes of this repository's workloads."""
import pytest
import torch

pytestmark = pytest.mark.gpu

F32, BF16 = torch.float32, torch.bfloat16


@pytest.mark.parametrize("B,L,d,dtype,pipelined,kernels", [
    (8, 4, 16, F32, False, ["k_chain"]),
    (256, 8, 3072, F32, False, ["k_chain"]),
    (256, 8, 3072, F32, True, ["k_tiles", "k_finish"]),
    (200, 8, 4096, F32, False, ["k_tiles", "k_finish"]),              # more than 300 KB a CTA
    (64, 16, 16384, BF16, False, ["k_tiles", "k_finish"]),
    (64, 16, 16384, BF16, True, ["k_tiles", "k_finish"]),
    (16, 32, 196608, F32, False, ["k_tiles", "k_finish_long"]),
    (16, 32, 196608, F32, True, ["k_tiles", "k_finish_long"]),
])
def test_kernels_of_a_call(B, L, d, dtype, pipelined, kernels):
    import __graft_entry__ as g
    g.build()
    import bench
    from paper_2606_13426_gb300 import api
    x = torch.zeros(B, L, d, dtype=dtype, device="cuda")
    sigma = torch.ones(L, device="cuda")
    ws = api.make_workspace(B, L, d, dtype)
    out = dict(accepted_len=torch.empty(B, dtype=torch.int32, device="cuda"),
               y=torch.empty(B, d, dtype=dtype, device="cuda"), status=torch.empty(B, dtype=torch.int32, device="cuda"))

    def call():
        api.verify(x, x, x, sigma, 1, "block", with_ratios=False, workspace=ws, out=out, pipelined=pipelined)
    call()
    torch.cuda.synchronize()
    assert bench.kernels_of_call(torch.cuda.Stream(), call) == kernels
