"""Form of deep FP64-accurate products where the scratch is small: a K panel that the scratch halves costs the residues
their splits and reconstructions again, so digits take over; both forms give the product."""
import ctypes

import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n,k,mb,residues", [
    (1024, 1024, 4096, 64, False), (1024, 1024, 4096, 128, False), (1024, 1024, 4096, 512, True),
    (2048, 2048, 4096, 128, False), (2048, 2048, 4096, 256, True), (300, 8000, 4096, 64, False),
    (3000, 3000, 9000, 128, False), (3000, 3000, 9000, 512, True)])
def test_form(m, n, k, mb, residues):
    import torch
    from paper_1504_06443_gb300 import build
    build.build()
    import paper_1504_06443_gb300 as gep
    g = torch.Generator(device="cuda").manual_seed(m + k)
    A = torch.randn(k, m, generator=g, dtype=torch.float64, device="cuda").t()
    B = torch.randn(n, k, generator=g, dtype=torch.float64, device="cuda").t()
    C = torch.empty(n, m, dtype=torch.float64, device="cuda").t()
    ws = torch.empty(mb << 20, dtype=torch.uint8, device="cuda")
    h = gep.Handle()
    ptr = lambda t: ctypes.c_void_p(t.data_ptr())
    assert h.lib.gep_set_workspace(h.h, ptr(ws), ws.numel()) == 0
    h.profile_enable(1000)
    assert h.lib.gep_dgemm(h.h, b"N", b"N", b"F", m, n, k, 1.0, ptr(A), m, ptr(B), k, 0.0, ptr(C), m, 1) == 0
    p = h.profile_read()
    h.profile_enable(0)
    h.close()
    # 16 plane products a residue product, 36 a digit product
    assert abs(p["tensor_flops"] / p["fp64_flops"] - (16 if residues else 36)) < 1e-6
    ref = A @ B
    assert float((C - ref).abs().max()) <= 4 * k * 2.0 ** -52 * float(A.abs().max() * B.abs().max())
