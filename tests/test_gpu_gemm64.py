"""FP64 products on the tensor cores at the edges of their tiles (128 x 64), stages (32
columns) and chunks (128): the density of H lattices against extended precision."""
import numpy as np
import pytest

import paper_2303_00689_gb300 as kx
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 3, 17, 31, 32, 33, 63, 64, 65, 127, 128, 129, 191, 193, 255, 257, 385])
def test_density_of_fp64_handles_is_the_rounded_product(n):
    side = int(np.ceil(n ** (1.0 / 3.0)))
    rng = np.random.default_rng(n)
    R = 1.9 * np.array([[i % side, i // side % side, i // side ** 2] for i in range(n)], dtype=float)
    R += 0.1 * rng.normal(size=R.shape)
    cfg = kx.sim_config_default(Te=5000.0, precision=kx.SIM_PREC_FP64, kernel=kx.SIM_KERNEL_XL)
    table = kx.param_table(synth.table_to_array(synth.synthetic_table(1)))
    Z = np.ones(n, dtype=np.int32)
    h = kx.sim_create(cfg, table, Z, R, V=synth.maxwell_boltzmann(Z, 300.0, seed=n), charge=n % 2,
                      P0=0.5 * (1.0 - (n % 2) / n) * np.eye(n))
    try:
        Q, D = kx.sim_get_matrix(h, kx.SIM_MAT_Q), kx.sim_get_matrix(h, kx.SIM_MAT_D0)
        f = kx.sim_get_vector(h, 1)
    finally:
        kx.sim_destroy(h)
    Qs = Q * np.sqrt(f)
    a = np.abs(Qs)
    exact = Qs.astype(np.longdouble) @ Qs.T.astype(np.longdouble)
    # Q f^1/2 in two roundings each; digits to 2^-63 of the row maximum, the kept products to
    # 2^-60 of their product a column; one rounding of the result
    tol = 2.0 ** -51 * (a @ a.T) + n * 2.0 ** -60 * np.outer(a.max(axis=1), a.max(axis=1))
    assert np.array_equal(D, D.T)
    assert (np.abs(D - exact) <= tol).all()
