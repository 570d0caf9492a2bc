"""FP32 preconditioner on levels that keep their stencil (at most 4,096 cells) and on the level just
above, walls and periodic, viscous, every agglomeration factor, single rows and columns of cells."""
from dataclasses import replace

import numpy as np
import pytest

import synth
from oracle.fv import Multigrid
from tests._common import gpu_context, oracle_dg, perturbed_state, rel, to_cpu, to_gpu

pytestmark = pytest.mark.gpu

W, V = synth.BUBBLE_Q2_20x10, synth.DENSITY_CURRENT_Q2_256x32
CASES = [
    ("Q1 32x32: 4,096 cells", replace(synth.scaled(W, 32, 32), k=1), "mg001111V"),
    ("Q1 33x32: above", replace(synth.scaled(W, 33, 32), k=1), "mg001111V"),
    ("Q2 by 3, odd", synth.scaled(W, 7, 5), "mg111222W"),
    ("Q4 by 5, row", replace(synth.scaled(W, 6, 1), k=4), "mg111111V"),
    ("Q3 column, periodic", replace(synth.scaled(W, 1, 4), k=3, periodic_x=True), "mg111111V"),
    ("viscous Q2", synth.scaled(V, 12, 6), "mg111211V"),
    ("viscous Q1 periodic", replace(synth.scaled(V, 6, 4), k=1, periodic_x=True), "mg112111W"),
]


@pytest.mark.parametrize("name,w,key", CASES, ids=[c[0] for c in CASES])
def test_against_oracle(name, w, key):
    """Relative 2e-3 to the FP64 oracle's Q^-1 r, the suite's bound for the FP32 form (the oracle's
    finite differences with the parity numerator c = 1e-2)."""
    import torch
    dg = oracle_dg(w)
    U = perturbed_state(w, dg)
    r = synth.random_perturbation(dg.shape[1:], 3)
    adt = 0.3 * w.dt
    ctx = gpu_context(w, precond_prec=32, mg_key=key, fv_levels=3)
    z = torch.empty(ctx.N, dtype=torch.float64, device="cuda")
    ctx.mg_precondition(to_gpu(U.ravel()), adt, to_gpu(r.ravel()), z)
    mg = Multigrid(dg, 3, key, fd_eps=1e-2)
    mg.linearize(U, adt)
    assert rel(to_cpu(z, dg.shape), mg.apply(r)) < 2e-3
