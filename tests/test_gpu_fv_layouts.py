"""FP32 preconditioner on levels above the stored stencils' 4,096 cells: the four-lanes-a-cell kernels
and the face-once tiles (both heights), inviscid and viscous, walls and periodic, agglomeration by 2, 3
and 5, ragged tiles, a BF16 coarsest level."""
from dataclasses import replace

import numpy as np
import pytest

import synth
from oracle.fv import Multigrid
from tests._common import gpu_context, oracle_dg, perturbed_state, rel, to_cpu, to_gpu

pytestmark = pytest.mark.gpu

W, V = synth.BUBBLE_Q2_20x10, synth.DENSITY_CURRENT_Q2_256x32
CASES = [
    ("Q3 18,432 + 4,608 cells", replace(synth.scaled(W, 48, 24), k=3), 3, 32),
    ("Q1 periodic, ragged", replace(synth.scaled(W, 101, 42), k=1, periodic_x=True), 2, 32),
    ("Q2 by 3", synth.scaled(W, 37, 31), 2, 32),
    ("Q4 by 5", replace(synth.scaled(W, 26, 17), k=4), 2, 32),
    ("viscous Q1", replace(synth.scaled(V, 98, 48), k=1), 3, 32),
    ("viscous Q2 by 3, periodic", replace(synth.scaled(V, 41, 18), periodic_x=True), 2, 32),
    ("Q3, BF16 coarsest of 4,608 cells", replace(synth.scaled(W, 48, 24), k=3), 2, 16),
]
LAYOUTS = [dict(fv_split_cells=1 << 30), dict(fv_split_cells=1, tile_fv=128), dict(fv_split_cells=1, tile_fv=256)]


@pytest.mark.parametrize("name,w,levels,prec", CASES, ids=[c[0] for c in CASES])
def test_layouts_agree(name, w, levels, prec):
    """Against the oracle's Q^-1 r 2e-3 (BF16 2e-2), the suite's bounds.  Against each other: an FP32
    product rounds terms alpha dt lambda times its direction, eight roundings deep, and an application
    chains some of them; where BF16 rounds what differs in the last bit it may take either neighbour
    (2^-8 of values that weigh less than a tenth)."""
    import torch
    key = "mg111211V"
    dg = oracle_dg(w)
    U = perturbed_state(w, dg)
    r = synth.random_perturbation(dg.shape[1:], 3)
    adt = 0.3 * w.dt
    out = []
    for lay in LAYOUTS:
        ctx = gpu_context(w, precond_prec=prec, mg_key=key, fv_levels=levels, **lay)
        assert all(a * b > 4096 for a, b in ctx.fv_levels()[:1])
        z = torch.empty(ctx.N, dtype=torch.float64, device="cuda")
        ctx.mg_precondition(to_gpu(U.ravel()), adt, to_gpu(r.ravel()), z)
        out.append(to_cpu(z, dg.shape))
    mg = Multigrid(dg, levels, key, fd_eps=1e-2)
    mg.linearize(U, adt)
    ref = mg.apply(r)
    n1 = w.k + 1
    lam = 2.0 * 350.0 * (w.nx * n1 / (w.x1 - w.x0) + w.nz * n1 / (w.z1 - w.z0))
    products = mg.stats["dg_calls"] + sum(mg.stats["fv_calls"])
    close = products * 8 * 2.0 ** -24 * (1.0 + adt * lam) if prec == 32 else 2.0 ** -8 * 0.1
    assert close < 1e-3 or prec == 16
    for z in out:
        assert rel(z, ref) < (2e-3 if prec == 32 else 2e-2)
        assert rel(z, out[0]) < close
