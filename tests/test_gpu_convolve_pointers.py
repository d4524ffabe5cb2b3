"""bem_convolve reads and writes device fields in place where it can: every
combination of host and device arrays, one buffer for both, and device fields on
an 8-byte boundary give the host call's result, bitwise."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(48, 20), (31, 33), (256, 64), (1040, 6)])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_pointer_kinds(bem_mod, cuda_ok, nx, ny, prec):
    import torch
    r = np.random.Generator(np.random.PCG64(7))
    p = r.random((ny, nx))
    with bem_mod.Handle(nx, ny, 0.01, 0.02, -0.3, 0.3) as h:
        ref = h.convolve(p, precision=prec)
        pd = torch.from_numpy(p).cuda()
        ud = torch.empty_like(pd)
        assert np.array_equal(h.convolve(pd, precision=prec, out=ud).cpu().numpy(), ref)
        un = np.empty_like(p)
        assert np.array_equal(h.convolve(pd, precision=prec, out=un), ref)
        assert np.array_equal(h.convolve(p, precision=prec, out=torch.empty_like(pd)).cpu().numpy(), ref)
        big = torch.zeros(2 * nx * ny + 3, dtype=torch.float64, device="cuda")  # odd offsets: 8-byte aligned
        po, uo = big[1:1 + nx * ny].view(ny, nx), big[nx * ny + 2:2 * nx * ny + 2].view(ny, nx)
        po.copy_(pd)
        torch.cuda.synchronize()
        got = h.convolve(po, precision=prec, out=uo).cpu().numpy()
        # the unaligned fields may take other launch shapes: FP32 rounds elsewhere
        tol = 0.0 if prec == "fp64" else 2e-6 * np.abs(ref).max()
        assert np.abs(got - ref).max() <= tol
        assert float(big[0]) == 0.0 and float(big[nx * ny + 1]) == 0.0 and float(big[-1]) == 0.0
        assert np.array_equal(h.convolve(pd, precision=prec, out=pd).cpu().numpy(), ref)  # in place
