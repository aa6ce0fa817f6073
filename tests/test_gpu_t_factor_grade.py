"""T factors of the back-transformation are formed with FP64-accurate products whatever the engine: in a first pass
on the FP32-grade engine (6 plane products each) they are the ones that take more planes."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,merges", [(250, False), (500, True), (1100, True)])
def test_t_factor_products(M, merges):
    import torch
    from paper_1504_06443_gb300 import build
    build.build()
    import paper_1504_06443_gb300 as gep
    g = torch.Generator(device="cuda").manual_seed(M)
    A = torch.randn(M, M, generator=g, dtype=torch.float64, device="cuda")
    A = A + A.t()
    B = torch.eye(M, dtype=torch.float64, device="cuda")
    h = gep.Handle()
    h.profile_enable(20000)
    w, Y, info = gep.solve(A, B, precision="mixed_refined", sep="1stage", refine_iters=-1, handle=h)
    p = h.profile_read()
    h.profile_enable(0)
    h.close()
    assert info == 0 and p["skipped"] == 0 and p["launches"] > 0
    # merges of 256 and more reflectors go to the tensor cores; narrower ones run on the FP64 units
    assert (p["tensor_flops"] > 6.0000001 * p["fp64_flops"]) == merges
    assert float((Y.t() @ Y - B).abs().max()) <= 1e-3
