"""The allocation-free entry point runs the context's own arithmetic: G and the
weight of given fields are the same bits (odd and ragged sizes, doped and
half-filled, one and several slices per stabilisation)."""
import numpy as np
import pytest

from paper_2303_13403_gb300 import pqmc, workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("spec,n_stab", [
    (workloads.honeycomb(2, U=4.0, dtau=0.1, two_theta=2.0, g=0.6, M_N=0.21), 1),
    (workloads.ChainSpec(kind=workloads.SQUARE, Lx=5, Ly=5, tp=-0.2, U=4.0, two_theta=2.0, g=0.3, n_up=11, n_dn=12), 5),
    (workloads.GUTZ_72[4.0], 10),
    (workloads.honeycomb(9, U=4.0, dtau=0.1, two_theta=2.0, g=0.6, M_N=0.21), 10),
])
def test_same_bits_as_a_context(spec, n_stab):
    import torch
    torch.cuda.set_device(0)
    N = spec.n_sites
    fields = workloads.random_fields(spec, 7)
    ctx = pqmc.Context([spec], prec=pqmc.FP64, seed=1, n_stab=n_stab)
    ctx.set_fields(fields)
    d_fields = torch.from_numpy(fields).to("cuda")
    d_G = torch.full((2, N, N), float("nan"), dtype=torch.float64, device="cuda")
    d_w = torch.full((4,), float("nan"), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    pqmc.green_noalloc(spec, n_stab, d_fields.data_ptr(), d_G.data_ptr(), d_w.data_ptr(),
                       torch.cuda.current_stream().cuda_stream)
    assert np.array_equal(d_G.cpu().numpy(), np.stack([ctx.green(0, 0), ctx.green(0, 1)]))
    assert np.array_equal(d_w.cpu().numpy(), ctx.weight())
    ctx.close()
