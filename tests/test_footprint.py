"""The device memory of a context, by which states are admitted: no more bytes than before the solver
kept its linearisation (restart 30), whatever the viscosity; on a GPU, what is allocated stays within
it, and steps whose buffers share memory match the oracle."""
from dataclasses import replace

import numpy as np
import pytest

import synth
from oracle.solver import implicit_step
from tests._common import gpu_context, initial_state, oracle_dg, to_cpu, to_gpu

ADMITTED = {   # nx, nz, precision: orders 1 to 4
    (160, 80, 64): (175541632, 381135232, 677024832, 1032552832),
    (160, 80, 32): (141297632, 304660832, 535914432, 819700832),
    (20, 10, 64): (3797968, 7018768, 11653360, 17213968),
    (20, 10, 32): (3266568, 5828568, 9453960, 13894968),
    (80, 3, 64): (4345152, 8216864, 13782816, 20464608),
    (80, 3, 32): (3717232, 6800264, 11157056, 16497208),
}


@pytest.mark.parametrize("nx,nz,prec", list(ADMITTED))
def test_admitted_as_before(nx, nz, prec):
    import paper_2505_24504_gb300 as P
    from paper_2505_24504_gb300 import build
    build.build()
    for k, most in enumerate(ADMITTED[nx, nz, prec], start=1):
        g = P.Grid(nx, nz, 0.0, 20000.0, 0.0, 10000.0, 0)
        assert P.Context.workspace_bytes(g, k, P.Opts.defaults(precond_prec=prec, fv_levels=5)) <= most, k


W, V = synth.BUBBLE_Q2_20x10, synth.DENSITY_CURRENT_Q2_256x32
OPTS = [dict(precond_prec=32), dict(precond_prec=32, dg_fused=2), dict(precond_prec=32, gmres_restart=1),
        dict(precond_prec=32, rk_stages=2, rk_alpha=(0.5, 1.0)), dict(precond_prec=16, mg_key=""),
        dict(precond_prec=64), dict(precond_prec=64, precond_fd_eps=1e-2, gmres_restart=40), dict(precond_prec=64, mg_key="")]


@pytest.mark.gpu
@pytest.mark.parametrize("opt", OPTS, ids=lambda o: " ".join(f"{k}={v}" for k, v in o.items()))
@pytest.mark.parametrize("w", [replace(synth.scaled(W, 160, 120), k=3), replace(synth.scaled(V, 160, 120), k=3)], ids=["Euler", "viscous"])
def test_allocations_stay_within(w, opt):
    """2 MiB an array for the allocator's granularity."""
    import paper_2505_24504_gb300 as P
    import torch
    torch.zeros(1, device="cuda")
    gpu_context(synth.scaled(W, 2, 2)).close()   # the library's own first allocations
    est = P.Context.workspace_bytes(P.Grid(w.nx, w.nz, w.x0, w.x1, w.z0, w.z1, 0), w.k,
                                    P.Opts.defaults(**dict(dict(fv_levels=w.fv_levels, mg_key=w.mg_key), **opt)))
    before = torch.cuda.mem_get_info()[0]
    ctx = gpu_context(w, **opt)
    used = before - torch.cuda.mem_get_info()[0]
    ctx.close()
    assert used <= est + 100 * (2 << 20), (used, est)


@pytest.mark.gpu
@pytest.mark.parametrize("restart", [1, 3, 17, 18])
@pytest.mark.parametrize("opt", [dict(precond_prec=64), dict(precond_prec=64, precond_fd_eps=1e-6), dict(precond_prec=32),
                                 dict(precond_prec=32, profile=1), dict(precond_prec=64, use_graphs=0),
                                 dict(precond_prec=32, mg_key="")],
                         ids=lambda o: " ".join(f"{k}={v}" for k, v in o.items()))
def test_restarted_steps(restart, opt):
    """Steps that restart on bases around the 16 vectors with float copies of their own: both solve to
    1e-8 of |G0|, so the increments agree to 1e-6 (the suite's bound)."""
    if opt.get("mg_key") == "" and restart < 17:
        pytest.skip("no convergence within 300 iterations without a preconditioner")
    w = replace(synth.scaled(W, 8, 6), k=3)
    dg = oracle_dg(w)
    U0 = initial_state(w, dg)
    ctx = gpu_context(w, gmres_restart=restart, **opt)
    U = to_gpu(U0.ravel())
    dt = w.dt * (0.25 if restart == 1 else 1.0)
    ctx.implicit_step(U, dt, scheme=1)
    ref = implicit_step(dg, U0, dt, scheme=1, tol=w.newton_tol)
    err = np.linalg.norm(to_cpu(U, dg.shape) - ref) / np.linalg.norm(ref - U0)
    assert err < 1e-6, err
