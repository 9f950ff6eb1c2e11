"""Stack blocks that the Cholesky QR cannot factorise.

With 2 Theta = 0 the stack blocks are e^{V(s)} P alone, formed in FP64, and a
large g makes them as ill-conditioned as wanted: the Gutzwiller factor scales
the sites of field +1 up (spin down: those of field -1) and the others down,
so a spin with fewer scaled-up sites than particles has a block with
cond ~ e^{2 kappa}, kappa = arccosh(e^{g/2}) (g = 18: 2.6e8), beyond the
1e6 that the factorisation takes.  The host decides which blocks break from
the fields; a block in between is left to neither side."""
import numpy as np
import pytest

from oracle import philox, pqmc as opq
from paper_2303_13403_gb300 import pqmc, workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def cuda():
    import torch
    torch.cuda.set_device(0)
    pqmc.load()


def vmc(L, g, **kw):
    return workloads.honeycomb(L, U=4.0, dtau=0.1, two_theta=0.0, g=g, M_N=0.21, **kw)


def model_of(spec):
    return opq.Model(opq.Params(kind=spec.kind, Lx=spec.Lx, Ly=spec.Ly, U=spec.U, dtau=spec.dtau, two_theta=spec.two_theta,
                                g=spec.g, M_N=spec.M_N, n_up=spec.n_up, n_dn=spec.n_dn, n_stab=1))


def smallest_pivot(m, fields, sg):
    """Smallest pivot of the blocks' Gram matrices relative to its diagonal (both end slices)."""
    out = 1.0
    for f in fields:
        M = np.exp(sg * np.arccosh(np.exp(m.p.g / 2)) * f)[:, None] * m.P[sg]
        r = np.abs(np.diag(np.linalg.qr(M)[1]))
        out = min(out, float((r ** 2 / (M ** 2).sum(0)).min()))
    return out


@pytest.mark.parametrize("prec", [pqmc.FP64, pqmc.FP32])
@pytest.mark.parametrize("L,g", [(3, 18.0), (6, 18.0), (6, 0.6)])
def test_spread_reports_a_breakdown(L, g, prec):
    """The whole-GPU sweep has no other factorisation: it stops with ESTAB, at
    whichever column the pivot fails, and the next context runs."""
    spec = vmc(L, g)
    m = model_of(spec)
    seen = set()
    for seed in range(1, 9):
        f = philox.initial_fields(seed, 0, 2, spec.n_sites)
        pivot = min(smallest_pivot(m, f, sg) for sg in (1, -1))
        if 2e-13 < pivot < 5e-12:
            continue
        try:
            pqmc.Context([spec], prec=prec, seed=seed, n_stab=1, spread=1).close()
            status = 0
        except pqmc.PQMCError as e:
            status = e.status
        assert status == (pqmc.ESTAB if pivot < 1e-12 else 0), (seed, pivot)
        seen.add(status)
    assert seen == {pqmc.ESTAB} if g > 1 else seen == {0}


def test_overflowing_exponential_is_reported():
    """e^{+dtau K} beyond the FP64 range (4 x 4, t' = -0.5: e^{720}, where
    e^{-dtau K} reaches e^{240}): the propagated G is NaN, which the first
    decisions taken on it report."""
    spec = workloads.ChainSpec(kind=workloads.SQUARE, Lx=4, Ly=4, tp=-0.5, U=0.0, dtau=120.0, two_theta=240.0, g=0.0,
                               n_up=7, n_dn=7)
    ctx = pqmc.Context([spec], prec=pqmc.FP64, seed=3, n_stab=1)
    with pytest.raises(pqmc.PQMCError) as e:
        ctx.sweep(2)
        ctx.synchronize()
    assert e.value.status == pqmc.ENAN
    ctx.close()


# (L, N_up, N_dn, sites of field +1): spin up breaks when these are fewer than N_up, spin down when the others
# are fewer than N_dn
BROKEN = [(3, 9, 9, 6), (3, 9, 9, 12), (3, 11, 11, 9), (6, 36, 36, 30), (6, 36, 36, 42), (6, 38, 38, 36), (6, 38, 34, 36),
          (6, 34, 38, 36), (9, 81, 81, 75), (9, 81, 81, 87)]


@pytest.mark.parametrize("prec", [pqmc.FP32, pqmc.BF16X3])
@pytest.mark.parametrize("tpb", [64, 256, 512])
@pytest.mark.parametrize("L,n_up,n_dn,plus", BROKEN)
def test_reduced_paths_fall_back_to_householder(L, n_up, n_dn, plus, tpb, prec):
    """One spin's block or both spins' beyond the Cholesky QR, in shared memory
    and (162 sites) global memory: G at tau = 0 and the weights of the FP64 path.
    Both end slices hold the same fields, so Q_L and Q_R span one space and G is
    1 minus a projector with elements of at most 1: three FP32 roundings and two
    sums of n terms, 2 (n + 3) 2^-24 = 1e-5 at n = 81."""
    spec = vmc(L, 18.0, n_up=n_up, n_dn=n_dn)
    rng = np.random.default_rng(plus)
    f = np.full(spec.n_sites, -1, np.int8)
    f[rng.permutation(spec.n_sites)[:plus]] = 1
    fields = np.stack([f, f])
    m = model_of(spec)
    for sg, broken in ((1, plus < n_up), (-1, spec.n_sites - plus < n_dn)):
        pivot = smallest_pivot(m, fields, sg)
        assert pivot < 1e-13 if broken else pivot > 1e-10
    out = []
    for p, threads in ((pqmc.FP64, 0), (prec, tpb)):
        ctx = pqmc.Context([spec], prec=p, seed=1, n_stab=1, cta_threads=threads)
        ctx.set_fields(fields)
        out.append(([ctx.green_at(0, 0, s) for s in (0, 1)], ctx.weight()))
        ctx.close()
    (G64, w64), (G, w) = out
    for s in (0, 1):
        assert np.abs(G64[s]).max() < 1 + 1e-6
        assert np.abs(G[s] - G64[s]).max() < 1e-5
    assert np.allclose(w, w64, rtol=0, atol=1e-6)
