"""The Krylov basis and Hessenberg columns of the solver's Arnoldi process: orthogonality and the
Arnoldi relation in FP64, also where the first Gram-Schmidt pass takes so little off the new vector
that the size test would leave the second one out."""
from dataclasses import replace

import pytest

import synth
from tests._common import gpu_context, oracle_dg, perturbed_state, to_gpu

pytestmark = pytest.mark.gpu

W = synth.BUBBLE_Q2_20x10
GRIDS = [(6, 5, 1), (9, 7, 2), (20, 10, 2), (33, 17, 3)]


def basis(nx, nz, k, nv):
    """nv columns without a preconditioner at 30 times the acoustic step, where the operator's skew
    part dominates and most columns leave more than the first pass takes off."""
    w = replace(synth.scaled(W, nx, nz), k=k)
    dg = oracle_dg(w)
    U = to_gpu(perturbed_state(w, dg).ravel())
    r = to_gpu(synth.random_perturbation(dg.shape[1:], 5).ravel())
    ctx = gpu_context(w, mg_key="", gmres_restart=32)
    V, H = ctx.arnoldi(U, 3.0 * w.dt, r, nv)
    return ctx, U, 3.0 * w.dt, V, H


def check(ctx, U, adt, V, H):
    """A dot product here is a chain of at most 64 FP64 roundings a thread and its trees, an update one
    of nv <= 32; four such sums enter an inner product of two normalised vectors: 4 (64 + 3 * 32) 2^-53
    = 7e-14, taken as 1e-13.  (A pass in FP32 alone leaves some 1e-8.)"""
    import torch
    nv = H.shape[1]
    gram = V @ V.T - torch.eye(nv + 1, dtype=torch.float64, device="cuda")
    assert float(gram.abs().max()) < 1e-13, float(gram.abs().max())
    for j in range(nv):
        w = torch.empty_like(U)
        ctx.jv_product(U, None, V[j].contiguous(), adt, 0.0, w)
        left = w - V.T @ to_gpu(H[:, j])
        assert float(left.norm() / w.norm()) < 1e-13, j


@pytest.mark.parametrize("nx,nz,k", GRIDS)
def test_single_precision_first_pass(nx, nz, k):
    """Columns against 1 to 16 vectors, whose first pass runs in FP32."""
    ctx, U, adt, V, H = basis(nx, nz, k, 16)
    assert any(H[j + 1, j] ** 2 > (H[:j + 1, j] ** 2).sum() for j in range(16))
    check(ctx, U, adt, V, H)


@pytest.mark.parametrize("nx,nz,k", GRIDS)
def test_long_basis(nx, nz, k):
    """Columns against 17 to 32 vectors as well (FP64 first pass, second pass by the size test)."""
    ctx, U, adt, V, H = basis(nx, nz, k, 32)
    assert any(H[j + 1, j] ** 2 > (H[:j + 1, j] ** 2).sum() for j in range(16, 32))
    check(ctx, U, adt, V, H)
