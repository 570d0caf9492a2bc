"""FP64 flux arithmetic at the edges of its ranges: the EOS power across its table
intervals and exponents, and states whose quotients and roots leave the fast range."""
import numpy as np
import pytest

from tests._common import gpu_context, oracle_dg, perturbed_state, to_cpu, to_gpu
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cp,cv", [(1005.0, 717.95), (1004.0, 717.0), (2000.0, 1000.0), (1300.0, 1000.0)])
def test_eos_power_at_interval_edges(cp, cv):
    """p = p0 (R E / p0)^gamma against numpy's long double at the edges of the 512 intervals and of
    the binary exponents, and outside the table (gamma = 2: c_3 = 0).  Tolerance: inside the table
    four half-ulp roundings; outside it CUDA's pow (2 ulp), the argument's two half-ulp roundings
    times gamma and the final product: 2.5 + gamma ulp."""
    import torch
    from dataclasses import replace
    w = replace(synth.scaled(synth.BUBBLE_Q2_20x10, 2, 2), cp=cp, cv=cv)
    ctx = gpu_context(w)
    m = 1.0 + np.arange(513) / 512.0
    m = np.concatenate([np.nextafter(m[1:], 0), m[:-1], np.nextafter(m[:-1], 2)])
    E = np.concatenate([np.ldexp(m, e) for e in (-40, -33, -32, -1, 0, 7, 8, 31, 32, 40)])
    x = to_gpu(E)
    p = torch.empty_like(x)
    ctx.eos_pressure(x, p)
    L = np.longdouble
    # the library's constants: R = cp - cv, gamma = cp / cv and (outside the table) R / p0 as doubles
    R, gam = cp - cv, cp / cv
    ref = L(w.p0) * (L(R) / L(w.p0) * E.astype(L)) ** L(gam)
    ulp = np.abs(to_cpu(p) - ref) / np.spacing(ref.astype(np.float64))
    assert float(ulp.max()) <= 2.5 + gam


@pytest.mark.parametrize("var,bad", [(0, np.nan), (0, np.inf), (3, -1.0e4)])
def test_unphysical_states_stay_non_finite(var, bad):
    """A NaN or infinite density or a negative rho theta reaches the residual as non-finite values
    in that element (no finite garbage from the fast quotients), and stays out of distant ones."""
    import torch
    w = synth.scaled(synth.BUBBLE_Q2_20x10, 4, 3)
    dg = oracle_dg(w)
    U = perturbed_state(w, dg)
    U[var, 1, 2, 1, 1] = bad
    ctx = gpu_context(w)
    f = torch.empty(ctx.N, dtype=torch.float64, device="cuda")
    ctx.dg_residual(to_gpu(U.ravel()), f)
    with np.errstate(all="ignore"):
        ref = dg.rhs(U)
    got = to_cpu(f, dg.shape)
    assert not np.isfinite(got[:, 1, 2]).all()
    assert not np.isfinite(ref[:, 1, 2]).all()
    assert np.isfinite(ref[:, 0, 0]).all() and np.isfinite(got[:, 0, 0]).all()
