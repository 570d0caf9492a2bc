"""The finite-difference product about a stored linearisation (what the solver's Arnoldi steps
use; jv_product takes it when it evaluates f(U) itself and eps is the default) against the
oracle's complex-step derivative and against the general form."""
from dataclasses import replace

import numpy as np
import pytest

import synth
from tests._common import gpu_context, oracle_dg, perturbed_state, rel, to_cpu, to_gpu

pytestmark = pytest.mark.gpu

W = synth.BUBBLE_Q2_20x10
CASES = [   # edges of the launch shapes: one element, ragged blocks, every order, periodic, viscous
    ("single Q1", replace(synth.scaled(W, 1, 1), k=1)),
    ("row Q4", replace(synth.scaled(W, 7, 1), k=4)),
    ("column Q3", replace(synth.scaled(W, 1, 5), k=3)),
    ("ragged Q1", replace(synth.scaled(W, 23, 9), k=1)),
    ("ragged Q2", replace(synth.scaled(W, 13, 11), k=2)),
    ("Q3", replace(synth.scaled(W, 16, 8), k=3)),
    ("Q4", replace(synth.scaled(W, 9, 7), k=4)),
    ("periodic Q3", synth.scaled(synth.INERTIA_GRAVITY_Q3_80x3, 10, 3)),
    ("viscous Q1", replace(synth.scaled(synth.DENSITY_CURRENT_Q2_256x32, 11, 5), k=1)),
    ("viscous Q2", synth.scaled(synth.DENSITY_CURRENT_Q2_256x32, 16, 4)),
    ("viscous Q3", replace(synth.scaled(synth.DENSITY_CURRENT_Q2_256x32, 6, 5), k=3)),
    ("viscous Q4 periodic", replace(synth.scaled(synth.DENSITY_CURRENT_Q2_256x32, 5, 4), k=4, periodic_x=True)),
]


@pytest.mark.parametrize("name,w", CASES, ids=[c[0] for c in CASES])
def test_product_about_linearisation(name, w):
    """Both forms carry the fluxes' rounding noise over eps; the stored form may not carry more
    (25 % allowed between two draws of the same noise), and both meet the 2e-3 of the paper's eps."""
    import torch
    dg = oracle_dg(w)
    U = perturbed_state(w, dg)
    y = synth.random_perturbation(dg.shape[1:], 11)
    adt = 0.3 * w.dt
    exact = dg.jv_exact(U, y, adt)
    for prec in (64, 32):
        ctx = gpu_context(w, precond_prec=prec)
        Ug, yg = to_gpu(U.ravel()), to_gpu(y.ravel())
        f, J1, J2 = (torch.empty_like(Ug) for _ in range(3))
        ctx.dg_residual(Ug, f)
        ctx.jv_product(Ug, f, yg, adt, 0.0, J1)          # general form
        ctx.jv_product(Ug, None, yg, adt, 0.0, J2)       # about the stored linearisation
        scale = np.linalg.norm((exact - y).ravel())      # the J part
        e1, e2 = (np.linalg.norm(to_cpu(J, dg.shape) - exact) / scale for J in (J1, J2))
        assert e2 <= 1.25 * e1 + 1e-9, (e1, e2)
        assert rel(to_cpu(J2, dg.shape), exact) < 2e-3
        z = torch.zeros_like(yg)
        ctx.jv_product(Ug, None, z, adt, 0.0, J2)
        assert float(J2.abs().max()) == 0.0              # y = 0
        z[3] = float("nan")
        ctx.jv_product(Ug, None, z, adt, 0.0, J2)
        assert not bool(torch.isfinite(J2).all())        # NaN is not swallowed


@pytest.mark.parametrize("e", [-330, -130, 130, 330])
def test_direction_of_any_magnitude(e):
    """eps is inversely proportional to |y|, so a direction scaled by a power of two gives the scaled
    product bit for bit (also far outside the range of single precision)."""
    import torch
    w = synth.scaled(synth.DENSITY_CURRENT_Q2_256x32, 9, 4)
    dg = oracle_dg(w)
    U, y = to_gpu(perturbed_state(w, dg).ravel()), to_gpu(synth.random_perturbation(dg.shape[1:], 11).ravel())
    ctx = gpu_context(w)
    J1, J2 = torch.empty_like(U), torch.empty_like(U)
    ctx.jv_product(U, None, y, 0.3 * w.dt, 0.0, J1)
    ctx.jv_product(U, None, y * 2.0 ** e, 0.3 * w.dt, 0.0, J2)
    assert bool(((J2 * 2.0 ** -e) == J1).all())
