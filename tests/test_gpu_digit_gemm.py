"""The FP64 products on the tensor cores (exact fixed-point digits) and the
phases built on them, at the sizes where they can go wrong.

Tolerance of a product: an element is rounded to 2^-62 of a power of two that
is at most twice the operand's largest element, the digit pairs left out stay
below 7 * 2^14 * 2^48 * (1 + 2^-7) of 2^124, so a term is off by at most 2^-57
max|A| max|B| (both effects), a sum of K terms by K times that, and the result
is rounded once.
"""
from dataclasses import replace

import numpy as np
import pytest

from oracle import pqmc as opq
from paper_2303_13403_gb300 import pqmc, workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def cuda():
    import torch
    torch.cuda.set_device(0)
    pqmc.load()


def product(A, B, strided):
    import torch
    dA, dB = torch.tensor(A, device="cuda"), torch.tensor(B, device="cuda")
    dC = torch.full((A.shape[0], B.shape[1]), 7.0, device="cuda", dtype=torch.float64)
    torch.cuda.synchronize()
    pqmc.test_digit_gemm(A.shape[0], B.shape[1], A.shape[1], dA.data_ptr(), dB.data_ptr(), dC.data_ptr(), strided)
    return dC.cpu().numpy()


@pytest.mark.parametrize("strided", [False, True])
@pytest.mark.parametrize("M,N,K", [(1, 1, 1), (16, 8, 16), (17, 9, 15), (36, 36, 72), (72, 72, 21), (33, 40, 128),
                                   (18, 7, 129), (20, 24, 648)])
def test_product_against_extended_precision(M, N, K, strided):
    rng = np.random.default_rng(M + 31 * N + 977 * K)
    for sa, sb in ((1.0, 1.0), (1e-150, 1e120)):
        A = sa * rng.standard_normal((M, K)) * 10.0 ** rng.uniform(-4, 0, (M, K))
        B = sb * rng.standard_normal((K, N))
        C = product(A, B, strided)
        ref = A.astype(np.longdouble) @ B.astype(np.longdouble)
        tol = K * 2.0 ** -56 * np.abs(A).max() * np.abs(B).max() + 2.0 ** -52 * np.abs(ref)
        assert np.all(np.abs(C - ref) <= tol)


def test_product_special_values():
    rng = np.random.default_rng(3)
    A, B = rng.standard_normal((20, 40)), rng.standard_normal((40, 12))
    assert np.array_equal(product(np.zeros_like(A), B, False), np.zeros((20, 12)))
    for bad in (np.nan, np.inf, -np.inf):
        X = A.copy()
        X[3, 5] = bad
        assert np.all(np.isnan(product(X, B, False)))
    # whole numbers: exact, signs and cancellation included
    A, B = rng.integers(-1000, 1000, (20, 40)).astype(float), rng.integers(-1000, 1000, (40, 12)).astype(float)
    assert np.array_equal(product(A, B, True), A @ B)


@pytest.mark.parametrize("prec,n_stab,tol", [(pqmc.FP64, 5, 1e-10), (pqmc.FP32, 1, 1e-4), (pqmc.FP32, 3, 1e-3)])
@pytest.mark.parametrize("Lx,Ly", [(2, 2), (3, 3), (5, 5), (9, 5)])
def test_green_at_every_stabilisation_point(prec, n_stab, tol, Lx, Ly):
    """Both stacks (odd numbers of products upwards among them), overlap, inverse
    and assembly at ragged sizes, against the oracle's definition."""
    spec = replace(workloads.honeycomb(2, U=4.0, two_theta=3.0 if n_stab != 3 else 2.4, g=0.3, M_N=0.21), Lx=Lx, Ly=Ly)
    fields = workloads.random_fields(spec, seed=5)
    ctx = pqmc.Context([spec], prec=prec, seed=5, n_stab=n_stab)
    ctx.set_fields(fields)
    m = opq.Model(opq.Params(kind=spec.kind, Lx=Lx, Ly=Ly, U=spec.U, dtau=spec.dtau, two_theta=spec.two_theta, g=spec.g,
                             M_N=spec.M_N, n_stab=n_stab, seed=5))
    for b in (0, 1, m.Ltau // n_stab):
        for s, sg in ((0, 1), (1, -1)):
            ref = opq.green_definition(m, fields, b * n_stab, sg)
            assert np.abs(ctx.green_at(b, 0, s) - ref).max() <= tol * max(1.0, np.abs(ref).max())


@pytest.mark.parametrize("delay_k", [8, 16, 32, 64])
def test_update_vectors_agree_over_cta_shapes(delay_k):
    """FP32 sweeps of 18, 72 and 98 sites (one and three lines short of whole
    vectors) with every CTA shape: the update vectors, decisions and products are
    the same sequences of FMAs, so accept logs and G agree exactly."""
    specs = [workloads.honeycomb(L, two_theta=0.8, g=0.6, M_N=0.21) for L in (3, 6, 7)]
    out = []
    for tpb, dense in ((64, 0), (128, 0), (256, 0), (512, 0), (64, 1), (128, 1)):
        ctx = pqmc.Context(specs, prec=pqmc.FP32, seed=4, n_stab=2, delay_k=delay_k, cta_threads=tpb, dense_chains=dense,
                           accept_log=1 << 14)
        ctx.sweep(2)
        out.append([(ctx.accept_log(2 * (s.n_slices + 2) * s.n_sites, c), ctx.green(c, 0), ctx.green(c, 1))
                    for c, s in enumerate(specs)])
        ctx.close()
    for o in out[1:]:
        for a, b in zip(out[0], o):
            assert all(np.array_equal(x, y) for x, y in zip(a, b))
