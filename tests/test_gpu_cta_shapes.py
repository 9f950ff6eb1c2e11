"""A chain's results do not depend on the CTA shape, which the default takes
from the number of chains in the context: accept logs, G, weights and the
records are the same bits with every shape, and a chain alone equals itself in a
batch of another default.  Ragged sizes (18, 25 and 72 sites), every delayed
block, both models."""
import numpy as np
import pytest

from paper_2303_13403_gb300 import pqmc, workloads

pytestmark = pytest.mark.gpu

HUBBARD = [workloads.honeycomb(3, two_theta=2.0, g=0.6, M_N=0.21),
           workloads.ChainSpec(kind=workloads.SQUARE, Lx=5, Ly=5, tp=-0.2, two_theta=2.0, g=0.3, n_up=11, n_dn=12),
           workloads.honeycomb(6, two_theta=2.0, g=0.6, M_N=0.21)]
TV = [workloads.tv_honeycomb(3, V=1.6, g=0.3, Delta_C=0.2, two_theta=2.0),
      workloads.tv_honeycomb(6, V=1.35, g=0.3, Delta_C=0.2, two_theta=2.0)]


@pytest.fixture(scope="module", autouse=True)
def cuda():
    import torch
    torch.cuda.set_device(0)
    pqmc.load()


def results(specs, tpb, dense=0, **kw):
    ctx = pqmc.Context(specs, cta_threads=tpb, dense_chains=dense, accept_log=1 << 14, **kw)
    ctx.sweep(2)
    out = []
    for c, s in enumerate(specs):
        species = 1 if s.kind == workloads.HONEYCOMB_TV else 2
        out.append([ctx.accept_log(2 * (s.n_slices + 2) * s.n_fields, c), ctx.weight(c), ctx.measurements(c)] +
                   [ctx.green(c, k) for k in range(species)])
    ctx.close()
    return out


def same(a, b):
    return all(np.array_equal(x, y) for p, q in zip(a, b) for x, y in zip(p, q))


@pytest.mark.parametrize("specs,delay_k", [(HUBBARD, 8), (HUBBARD, 16), (HUBBARD, 32), (HUBBARD, 64), (TV, 32)])
def test_fp64_shapes(specs, delay_k):
    ref = results(specs, 256, prec=pqmc.FP64, seed=6, n_stab=5, delay_k=delay_k)
    for tpb in (64, 128):
        assert same(ref, results(specs, tpb, prec=pqmc.FP64, seed=6, n_stab=5, delay_k=delay_k)), tpb


@pytest.mark.parametrize("specs", [HUBBARD, TV])
def test_fp32_shapes(specs):
    ref = results(specs, 256, prec=pqmc.FP32, seed=6, n_stab=2)
    for tpb, dense in ((64, 0), (128, 0), (512, 0), (64, 1), (128, 1)):
        assert same(ref, results(specs, tpb, dense, prec=pqmc.FP32, seed=6, n_stab=2)), (tpb, dense)


@pytest.mark.parametrize("chains", [200, 400])
def test_fp64_chain_alone_equals_itself_in_a_batch(chains):
    """One chain takes 256 threads by default, 200 take 128 and 400 take 64 (152 SMs)."""
    spec = workloads.honeycomb(3, two_theta=2.0, g=0.6, M_N=0.21)
    one = pqmc.Context([spec], prec=pqmc.FP64, seed=6, n_stab=5)
    batch = pqmc.Context([spec] * chains, prec=pqmc.FP64, seed=6, n_stab=5)
    assert one.launch()["cta_threads"] > batch.launch()["cta_threads"]
    one.sweep(3)
    batch.sweep(3)
    assert np.array_equal(one.measurements(0), batch.measurements(0))
    assert np.array_equal(one.green(0, 0), batch.green(0, 0))
    one.close()
    batch.close()
