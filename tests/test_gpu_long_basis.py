"""Arnoldi columns against 17 to 32 basis vectors (run-time basis size) and beyond 32 (general
multi-dot path): unpreconditioned steps whose linear solves need that many, on vectors whose
lengths leave ragged last blocks."""
from dataclasses import replace

import numpy as np
import pytest

import synth
from oracle.solver import implicit_step
from tests._common import gpu_context, initial_state, oracle_dg, to_cpu, to_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,nz,k,restart", [(6, 5, 1, 30), (7, 3, 2, 32), (9, 7, 2, 48), (11, 9, 3, 30)])
def test_unpreconditioned_step(nx, nz, k, restart):
    """One backward-Euler step against the oracle (modified Gram-Schmidt): both solve to 1e-8 of
    |G0|, so the increments agree to 1e-6 (the suite's bound), with the basis growing past 16."""
    w = replace(synth.scaled(synth.BUBBLE_Q2_20x10, nx, nz), k=k)
    dg = oracle_dg(w)
    U0 = initial_state(w, dg)
    ctx = gpu_context(w, mg_key="", gmres_restart=restart)
    U = to_gpu(U0.ravel())
    st = ctx.implicit_step(U, w.dt, scheme=0)
    assert st.gmres_its > 17 * st.newton_its / 2
    ref = implicit_step(dg, U0, w.dt, scheme=0, tol=w.newton_tol)
    err = np.linalg.norm(to_cpu(U, dg.shape) - ref) / np.linalg.norm(ref - U0)
    assert err < 1e-6, err
