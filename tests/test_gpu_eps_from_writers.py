"""FP64 preconditioner whose FD steps eps come from the kernels that wrote the directions: every
order of smoothing steps that hands an eps on or leaves it out, single cells, agglomeration by 2, 3
and 5, and a grid with more transfer blocks than partial sums (eps by a dot product)."""
from dataclasses import replace

import numpy as np
import pytest

import synth
from oracle.fv import Multigrid
from tests._common import gpu_context, oracle_dg, perturbed_state, rel, to_cpu, to_gpu

pytestmark = pytest.mark.gpu

C_FD = 1e-2
W, V = synth.BUBBLE_Q2_20x10, synth.DENSITY_CURRENT_Q2_256x32
CASES = [
    ("no smoothing before", replace(synth.scaled(W, 8, 4), k=1), "mg010101V", 3),
    ("none after", replace(synth.scaled(W, 8, 4), k=3), "mg101010W", 3),
    ("two of each", replace(synth.scaled(W, 6, 4), k=3), "mg222222V", 3),
    ("uneven, cycled", synth.scaled(W, 7, 5), "mg120221W", 3),
    ("no middle step before", replace(synth.scaled(W, 6, 4), k=1), "mg111101V", 3),
    ("one level", synth.scaled(W, 5, 3), "mg111211V", 1),
    ("by 5, one row", replace(synth.scaled(W, 6, 1), k=4), "mg111111W", 3),
    ("one element", replace(synth.scaled(W, 1, 1), k=1, periodic_x=True), "mg111111V", 2),
    ("viscous, odd", synth.scaled(V, 9, 5), "mg111111V", 2),
    ("4,097 transfer blocks", replace(synth.scaled(W, 241, 85), k=4), "mg111111V", 2),
]


@pytest.mark.parametrize("name,w,key,levels", CASES, ids=[c[0] for c in CASES])
def test_against_oracle(name, w, key, levels):
    """The rounding of f(u + eps y) weighs 2^-44 400 sqrt(n) / C_FD in a product of relative size one
    (eps |y_i| is about C_FD / sqrt(n)): that, times the products of the application, bounds the
    difference to the oracle; 1e-6 up to 1e5 unknowns, the suite's bar.  A second application gives
    the same bits (the reductions leave their counter as they found it)."""
    import torch
    dg = oracle_dg(w)
    U = perturbed_state(w, dg)
    r = synth.random_perturbation(dg.shape[1:], 5)
    adt = 0.3 * w.dt * min(1.0, 20.0 / w.nx)
    ctx = gpu_context(w, precond_prec=64, mg_key=key, fv_levels=levels, precond_fd_eps=C_FD)
    z, z2 = (torch.empty(ctx.N, dtype=torch.float64, device="cuda") for _ in range(2))
    ctx.mg_precondition(to_gpu(U.ravel()), adt, to_gpu(r.ravel()), z)
    ctx.mg_precondition(to_gpu(U.ravel()), adt, to_gpu(r.ravel()), z2)
    mg = Multigrid(dg, levels, key, fd_eps=C_FD)
    mg.linearize(U, adt)
    ref = mg.apply(r)
    products = mg.stats["dg_calls"] + sum(mg.stats["fv_calls"])
    bound = products * 2.0 ** -44 * 400.0 * np.sqrt(ctx.N) / C_FD + 1e-12
    assert rel(to_cpu(z, dg.shape), ref) < (min(1e-6, bound) if ctx.N <= 1e5 else bound)
    assert torch.equal(z, z2)
