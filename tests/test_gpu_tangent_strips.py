"""The fused FP32 tangent product at the edges of its strips: element counts around the strip
length of each order (21, 13, 8, 5 elements), single columns and rows, walls and periodic."""
from dataclasses import replace

import numpy as np
import pytest

import synth
from tests._common import gpu_context, oracle_dg, perturbed_state, to_cpu, to_gpu

pytestmark = pytest.mark.gpu

STRIP = {1: 21, 2: 13, 3: 8, 4: 5}
CASES = [(k, nx, nz, per) for k, e in STRIP.items()
         for nx, nz, per in ((1, 3, False), (e - 1, 2, True), (e, 1, False), (e + 1, 3, True), (2 * e + 1, 2, False))]


@pytest.mark.parametrize("k,nx,nz,per", CASES)
def test_strip_edges(k, nx, nz, per):
    """y - alpha dt J(U) y against the oracle's complex step, 2e-3 of the J part (the suite's bound for
    the FP32 product), and against the face + volume form to 1e-4."""
    import torch
    w = replace(synth.scaled(synth.BUBBLE_Q2_20x10, nx, nz), k=k, periodic_x=per)
    dg = oracle_dg(w)
    U = perturbed_state(w, dg)
    y = synth.random_perturbation(dg.shape[1:], 5)
    adt = 0.3 * w.dt
    exact = dg.jv_exact(U, y, adt)
    scale = np.linalg.norm((exact - y).ravel())
    outs = []
    for fused in (1, 2):
        ctx = gpu_context(w, precond_prec=32, dg_fused=fused)
        out = torch.empty(ctx.N, dtype=torch.float64, device="cuda")
        ctx.tangent_product(to_gpu(U.ravel()), to_gpu(y.ravel()), adt, out)
        outs.append(to_cpu(out, dg.shape))
        assert np.linalg.norm((outs[-1] - exact).ravel()) < 2e-3 * scale
    assert np.linalg.norm((outs[0] - outs[1]).ravel()) < 1e-4 * scale
