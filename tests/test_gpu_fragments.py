"""FP64 density between two fragments far apart: the products on the tensor cores are exact to 2^-60 of
the row maxima a column, whatever the size of the element, and that is below what the
eigenvectors' own rounding (2^-53) leaves in it."""
import numpy as np
import pytest

import paper_2303_00689_gb300 as kx
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [32, 80, 300])
@pytest.mark.parametrize("gap", [8.0, 14.0, 40.0])
def test_elements_between_fragments(n, gap):
    m = n // 2
    side = int(np.ceil(m ** (1.0 / 3.0)))
    P = 1.9 * np.array([[i % side, i // side % side, i // side ** 2] for i in range(m)], dtype=float)
    R = np.concatenate([P, P + [gap + 1.9 * (side - 1), 0.0, 0.0]])
    R += 0.1 * np.random.default_rng(n).normal(size=R.shape)
    cfg = kx.sim_config_default(Te=5000.0, precision=kx.SIM_PREC_FP64, kernel=kx.SIM_KERNEL_XL)
    table = kx.param_table(synth.table_to_array(synth.synthetic_table(1)))
    h = kx.sim_create(cfg, table, np.ones(n, dtype=np.int32), R, P0=0.5 * np.eye(n))
    try:
        Q, D, F = kx.sim_get_matrix(h, kx.SIM_MAT_Q), kx.sim_get_state(h, n)[3], kx.sim_get_matrix(h, kx.SIM_MAT_FOCK)
        f = kx.sim_get_vector(h, 1)
    finally:
        kx.sim_destroy(h)
    # the product: two roundings of Q f^1/2 and one of the result, and 2^-60 of the row maxima a column
    Qs = Q * np.sqrt(f)
    a = np.abs(Qs)
    exact = Qs.astype(np.longdouble) @ Qs.T.astype(np.longdouble)
    top = a.max(axis=1)
    assert (np.abs(D - exact) <= 2.0 ** -51 * (a @ a.T) + n * 2.0 ** -60 * np.outer(top, top)).all()
    # the element: LAPACK's eigenvectors, good to a few n 2^-53 in a density of norm one
    w, U = np.linalg.eigh(F)
    lo, hi = w[0] - 50.0, w[-1] + 50.0
    kT = 8.617333262e-5 * 5000.0
    for _ in range(200):
        mu = 0.5 * (lo + hi)
        occ = 1.0 / (1.0 + np.exp(np.clip((w - mu) / kT, -700.0, 700.0)))
        lo, hi = (mu, hi) if occ.sum() < n // 2 else (lo, mu)
    ref = (U * occ) @ U.T
    assert np.abs(D[:m, m:] - ref[:m, m:]).max() <= n * 2.0 ** -50
