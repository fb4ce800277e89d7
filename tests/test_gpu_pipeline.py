"""GPU parity of bistoch_normalize and eig_topk (FP64) against the oracle's
Algorithm 1 (Householder QR route), and end to end against the dense P (-m gpu).

Tolerances (FP64 path): degree vectors and Gram matrices 1e-12 relative,
eigenvalues 1e-10 relative, eigenvector subspaces (clusters of eigenvalues with
relative gap < 1e-6 compared as subspaces) 1e-8 in the sine of the largest
principal angle.
"""
import numpy as np
import pytest
import torch

from datagen import make_config
from oracle.pchol import greedy_pchol, arpc
from oracle.alg1 import bistochastic_evd, degree_vectors
from oracle.kernel import kernel_dense
from oracle.dense import bistochastic_dense, top_eigh
from tests.helpers import compare_eigpairs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def kevd():
    from paper_2510_26574_gb300.build import build
    build()
    import paper_2510_26574_gb300 as m
    return m


def _Fgpu(F):
    return torch.from_numpy(np.ascontiguousarray(F.T)).cuda()


def _check_normalize(kevd, F):
    rank = F.shape[1]
    dt, qt, A, C = kevd.bistoch_normalize(_Fgpu(F), rank)
    d0, q0 = degree_vectors(F)
    assert np.max(np.abs(dt.cpu().numpy() - d0) / np.abs(d0)) < 1e-12
    assert np.max(np.abs(qt.cpu().numpy() - q0) / np.abs(q0)) < 1e-12
    A0 = F.T @ (F / (d0 * d0)[:, None])
    C0 = F.T @ (F / q0[:, None])
    A = A.cpu().numpy()
    C = C.cpu().numpy()
    assert np.array_equal(A, A.T) and np.array_equal(C, C.T)
    assert np.max(np.abs(A - A0)) < 1e-12 * np.max(np.abs(A0))
    assert np.max(np.abs(C - C0)) < 1e-12 * np.max(np.abs(C0))
    return dt, qt


@pytest.mark.parametrize("case", ["ks2k_greedy", "arpc_ragged"])
def test_normalize_and_eig_match_alg1(kevd, case):
    if case == "ks2k_greedy":
        X, eps, _ = make_config("ks2k")
        F = greedy_pchol(X, eps, 128)[0]
        k = 32
    else:
        X, eps, _ = make_config("ks200k", N=3001)
        F = arpc(X, eps, 200, 40, 21)["F"]
        k = 40
    rank = F.shape[1]
    Fg = _Fgpu(F)
    dt, qt, A, C = kevd.bistoch_normalize(Fg, rank)
    _check_normalize(kevd, F)
    ev, U, kept = kevd.eig_topk(Fg, rank, dt, A, C, k)
    lam0, U0 = bistochastic_evd(F)
    ev = ev.cpu().numpy()
    U = U.cpu().numpy().T
    assert np.all(np.diff(ev) <= 0)
    erel, ang = compare_eigpairs(lam0[:k], U0[:, :k], ev, U, rel_gap=1e-6, lam_full=lam0)
    assert erel < 1e-10, erel
    assert ang < 1e-8, ang
    assert np.max(np.abs(U.T @ U - np.eye(k))) < 1e-10
    # sign convention: entry of largest magnitude is positive
    idx = np.argmax(np.abs(U), axis=0)
    assert np.all(U[idx, np.arange(k)] > 0)


def test_ks2k_end_to_end_vs_dense_P(kevd):
    """Config 1: greedy r=128 -> top-32 of P~, checked against the dense P."""
    X, eps, _ = make_config("ks2k")
    Xg = torch.from_numpy(X).cuda()
    out = kevd.rpchol_factor(Xg, eps, 128, mode="greedy")
    dt, qt, A, C = kevd.bistoch_normalize(out["F"], out["rank"])
    ev, U, kept = kevd.eig_topk(out["F"], out["rank"], dt, A, C, 32)
    ev = ev.cpu().numpy()
    P, _, _ = bistochastic_dense(kernel_dense(X, eps))
    lamP, UP = top_eigh(P, 32)
    # approximation error of the method (not parity): the leading eigenvalues agree closely
    assert abs(ev[0] - 1.0) < 1e-8 and abs(lamP[0] - 1.0) < 1e-12
    assert np.max(np.abs(ev[:8] - lamP[:8])) < 1e-3
    # Theorem 4 holds for this factor
    from oracle.bounds import theorem4_bound
    F = out["F"].cpu().numpy().T
    a, b = theorem4_bound(kernel_dense(X, eps), F @ F.T)
    assert a <= b


def test_degree_not_positive(kevd):
    # rows 0 and 2 of F F^T sum to zero
    F = np.array([[1.0, 0.0], [0.0, 1.0], [-1.0, 0.0]] + [[0.0, 1.0]] * 5)
    with pytest.raises(kevd.KevdError) as e:
        kevd.bistoch_normalize(_Fgpu(F), 2)
    assert e.value.status == 2


# FP64 Grams: with an even leading dimension (and F 16-byte aligned) the
# tensor-core kernel with exact digit-sliced products (gram_oz.cu) runs; an odd
# one, or KEVD_GRAM=fp64, the FP64-pipe kernel.  N = 3001 and 20,037 end in a
# partial 16-row quarter; rank 129 / 300 / 700 span several 128 x 64 tiles and
# leave ragged ones.
@pytest.mark.parametrize("N,rank,pad,gram", [(3001, 200, 1, None), (20000, 300, 0, None), (5000, 129, 3, None),
                                             (20037, 300, 1, None), (20000, 300, 0, "fp64"),
                                             (60000, 700, 0, None)])
def test_fp64_grams_tensor_core_and_fp64_pipe(kevd, monkeypatch, N, rank, pad, gram):
    """Both Gram matrices of an FP64 factor at the FP64 bar (1e-12 of the largest
    entry, exactly symmetric), and the one-Gram symmetric form."""
    if gram:
        monkeypatch.setenv("KEVD_GRAM", gram)
    X, eps, _ = make_config("ks200k" if rank < 500 else "vsa2m", N=N)
    F = arpc(X.astype(np.float64), eps, rank, 16 if rank < 500 else 100, 7)["F"]
    rk = F.shape[1]
    Fbuf = torch.full((rk, N + pad), float("nan"), dtype=torch.float64)
    Fbuf[:, :N] = torch.from_numpy(np.ascontiguousarray(F.T))
    Fg = Fbuf.cuda()[:, :N]
    dt, qt, A, C = kevd.bistoch_normalize(Fg, rk)
    d0, q0 = degree_vectors(F)
    A0 = F.T @ (F / (d0 * d0)[:, None])
    C0 = F.T @ (F / q0[:, None])
    A = A.cpu().numpy()
    C = C.cpu().numpy()
    assert np.array_equal(A, A.T) and np.array_equal(C, C.T)
    assert np.max(np.abs(A - A0)) < 1e-12 * np.max(np.abs(A0))
    assert np.max(np.abs(C - C0)) < 1e-12 * np.max(np.abs(C0))
    for G, G0 in ((A, A0), (C, C0)):
        assert abs(np.mean((np.diag(G) - np.diag(G0)) / np.diag(G0))) < 1e-13
    ds, As = kevd.symmetric_normalize(Fg, rk)
    As0 = F.T @ (F / d0[:, None])
    As = As.cpu().numpy()
    assert np.array_equal(As, As.T)
    assert np.max(np.abs(As - As0)) < 1e-12 * np.max(np.abs(As0))


# F views whose columns are not 16-byte aligned (odd leading dimension, or a start one
# element in): the Grams from seven digit planes.  Rank 65 / 129 leave one column in the
# last 64- and 128-column tile, N = 255 / 257 / 33 end inside and just past a 256-row
# chunk and a 32-row stage, N = 70,001 needs two row splits.  Bar: the operands carry
# 2^-55 of their column's largest entry, well inside the 1e-12 of the aligned layouts.
@pytest.mark.parametrize("N,rank,ld,off", [(255, 65, 255, 0), (257, 129, 261, 0), (33, 16, 33, 0), (4097, 64, 4098, 1),
                                           (70001, 130, 70001, 0)])
def test_fp64_grams_unaligned_layouts(kevd, N, rank, ld, off):
    g = torch.Generator().manual_seed(N)
    F = torch.rand(rank, N, generator=g, dtype=torch.float64) * torch.logspace(0, -3, rank, dtype=torch.float64)[:, None]
    buf = torch.full((rank * ld + off,), float("nan"), dtype=torch.float64, device="cuda")
    Fg = buf[off:].view(rank, ld)[:, :N]
    Fg.copy_(F)
    dt, qt, A, C = kevd.bistoch_normalize(Fg, rank)
    d0 = F.sum(1) @ F
    q0 = (F @ (1 / d0)) @ F
    for G, w in ((A, 1 / (d0 * d0)), (C, 1 / q0)):
        G0 = (F * w) @ F.T
        G = G.cpu()
        assert torch.equal(G, G.T)
        assert torch.max(torch.abs(G - G0)) < 1e-12 * torch.max(torch.abs(G0))


def test_fp64_grams_wide_weights(kevd):
    """Rows whose degree is 1e-25 of the others' (weights 1e50, beyond FP32's range) and an
    infinite entry: the first is within the bar of the FP64 sums, the second never comes
    out as a finite Gram."""
    N, rank = 3001, 40
    g = torch.Generator().manual_seed(5)
    F = torch.rand(rank, N, generator=g, dtype=torch.float64)
    F[:, 7] *= 1e-25
    Fg = F.cuda()
    dt, qt, A, C = kevd.bistoch_normalize(Fg, rank)
    d0 = F.sum(1) @ F
    A0 = (F / (d0 * d0)) @ F.T
    assert torch.max(torch.abs(A.cpu() - A0)) < 1e-12 * torch.max(torch.abs(A0))
    Fg[3, 11] = float("inf")
    try:
        _, _, A, C = kevd.bistoch_normalize(Fg, rank)
    except kevd.KevdError:
        return
    assert not torch.isfinite(A).all()


# A slab of the lift is bounded by the grid that cuts its planes (65,535 x 32 rows): at a small rank
# one more row than that takes two slabs.  The FP64 lift against the FP64-pipe GEMM with the bar of
# test_tensor_core_lift_matches_fp64_pipe, the FP32 one (three digits, 2^-22 of a row's largest
# entry in both factors, rank terms) against the same product of its F.
@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
def test_lift_more_rows_than_a_grid(kevd, monkeypatch, dtype):
    N, r, k = 65535 * 32 + 133, 8, 3
    g = torch.Generator(device="cuda").manual_seed(3)
    F = torch.rand(r, N, generator=g, dtype=dtype, device="cuda")
    d, q, A, C = kevd.bistoch_normalize(F, r)
    ev, U, kept = kevd.eig_topk(F, r, d, A, C, k)
    monkeypatch.setenv("KEVD_LIFT", "fp64")
    ev0, U0, _ = kevd.eig_topk(F.double(), r, d, A, C, k)
    assert torch.equal(ev, ev0) and kept == r
    bar = 1e-11 if dtype == torch.float64 else 16 * r * 2.0 ** -22
    scale = U0.abs().amax(1, keepdim=True)
    if dtype == torch.float32:      # entries of Y above 1 cancel in U
        R = torch.linalg.cholesky(A).T
        scale = torch.linalg.inv(R).abs().max() * F.max().double() / d.min()
    assert ((U - U0).abs() / scale).max().item() < bar
