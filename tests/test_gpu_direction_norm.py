"""eps of an Arnoldi step's product from the norm of what the FP32 preconditioner wrote: directions
whose squares overflow single precision within a block but not within a thread."""
from dataclasses import replace

import numpy as np
import pytest

import synth
from tests._common import gpu_context, oracle_dg, perturbed_state, to_gpu

pytestmark = pytest.mark.gpu

W = synth.BUBBLE_Q2_20x10
CASES = [("Q%d" % k, replace(synth.scaled(W, 24, 6), k=k)) for k in (1, 2, 3, 4)]
CASES.append(("viscous Q2", synth.scaled(synth.DENSITY_CURRENT_Q2_256x32, 24, 6)))


@pytest.mark.parametrize("name,w", CASES, ids=[c[0] for c in CASES])
def test_column_of_a_large_direction(name, w):
    """With one DG smoothing step as the preconditioner, z = sigma dtau r: sigma = 2^e scales the
    direction and its Hessenberg column exactly and leaves the next basis vector alone.  Single
    precision in the traces and the sum of squares bounds the difference by some 2^-23; 1e-5 allows
    for the product's own noise (the scaled eps is rounded to 24 bits in its linear terms)."""
    dg = oracle_dg(w)
    U = to_gpu(perturbed_state(w, dg).ravel())
    rng = np.random.default_rng(3)
    r = to_gpu(rng.choice([-1.0, 1.0], dg.shape).ravel() / np.sqrt(4 * dg.X.size))
    adt = 0.3 * w.dt
    opt = dict(precond_prec=32, mg_key="mg010000V", fv_levels=1)
    ctx = gpu_context(w, **opt)
    V, H = ctx.arnoldi(U, adt, r, 1)
    z = r.clone()
    ctx.mg_precondition(U, adt, r, z)
    node = 4 * float((z * z).mean())              # a thread's sum of squares
    nt = (w.k + 1) ** 2 * {1: 21, 2: 13, 3: 8, 4: 5}[w.k]   # nodes of a block
    e = int(round(0.5 * (130 - np.log2(node * nt))))
    assert 4 * float((z * z).max()) * 4.0 ** e < 2.0 ** 127 and node * nt * 4.0 ** e > 2.0 ** 128
    ctx = gpu_context(w, sigma_dg=2.0 ** e, **opt)
    V2, H2 = ctx.arnoldi(U, adt, r, 1)
    assert abs(H2 * 2.0 ** -e - H).max() < 1e-5 * abs(H).max()
    assert float((V2 - V).abs().max()) < 1e-5 * float(V.abs().max())
