"""Eigenvectors of degenerate levels: identical H2 molecules far apart, whose two levels
are clusters of as many members as there are molecules."""
import numpy as np
import pytest

import paper_2303_00689_gb300 as kx
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [kx.SIM_PREC_FP64, kx.SIM_PREC_MIXED])
@pytest.mark.parametrize("molecules", [1, 2, 3, 32, 33, 34, 65, 130])
def test_vectors_of_a_cluster_are_orthogonal(molecules, precision):
    side = int(np.ceil(molecules ** (1.0 / 3.0)))
    at = 400.0 * np.array([[i % side, i // side % side, i // side ** 2] for i in range(molecules)], dtype=float)
    R = np.concatenate([at[:, None, :], at[:, None, :] + [0.8, 0.0, 0.0]], axis=1).reshape(-1, 3)
    n = 2 * molecules
    cfg = kx.sim_config_default(Te=5000.0, precision=precision, kernel=kx.SIM_KERNEL_XL)
    table = kx.param_table(synth.table_to_array(synth.synthetic_table(1)))
    Z = np.ones(n, dtype=np.int32)
    h = kx.sim_create(cfg, table, Z, R, V=synth.maxwell_boltzmann(Z, 300.0, seed=1), P0=0.5 * np.eye(n))
    try:
        F, Q = kx.sim_get_matrix(h, kx.SIM_MAT_FOCK), kx.sim_get_matrix(h, kx.SIM_MAT_Q)
        eps = kx.sim_get_vector(h, 0)
    finally:
        kx.sim_destroy(h)
    width = max(1.0, np.abs(eps).max())
    # the tolerances of single levels: FP64, or 4-slice products (2^-24 of sum |a||b|)
    tol = 1e-6 if precision else 1e-10
    assert np.abs(Q.T @ Q - np.eye(n)).max() <= tol
    assert np.abs(F @ Q - Q * eps).max() <= tol * width * 10
