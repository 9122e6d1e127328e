"""Eigenvectors of nearly degenerate levels: H2 molecules far apart whose bonds differ by little, so
that the gaps within a cluster lie between the rounding of an eigenvalue and the cluster's tolerance."""
import numpy as np
import pytest

import paper_2303_00689_gb300 as kx
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [kx.SIM_PREC_FP64, kx.SIM_PREC_MIXED])
@pytest.mark.parametrize("molecules", [2, 9, 33, 70])
@pytest.mark.parametrize("step", [3e-13, 1e-12, 1e-11, 1e-10, 1e-9, 1e-8, 1e-7])
def test_vectors_of_a_near_cluster_are_orthogonal(molecules, step, precision):
    side = int(np.ceil(molecules ** (1.0 / 3.0)))
    at = 400.0 * np.array([[i % side, i // side % side, i // side ** 2] for i in range(molecules)], dtype=float)
    bond = 0.8 + step * np.arange(molecules)[:, None] * np.array([1.0, 0.0, 0.0])
    bond[:, 1:] = 0.0
    R = np.concatenate([at[:, None, :], (at + bond)[:, None, :]], axis=1).reshape(-1, 3)
    n = 2 * molecules
    cfg = kx.sim_config_default(Te=5000.0, precision=precision, kernel=kx.SIM_KERNEL_XL)
    table = kx.param_table(synth.table_to_array(synth.synthetic_table(1)))
    h = kx.sim_create(cfg, table, np.ones(n, dtype=np.int32), R, P0=0.5 * np.eye(n))
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
