"""Tridiagonalisation at the edges of its launch shapes: eigenpairs of the Fock matrix
of H lattices (one orbital per atom, so any n) against LAPACK, both precisions."""
import threading

import numpy as np
import pytest

import paper_2303_00689_gb300 as kx
import synth

pytestmark = pytest.mark.gpu


def _handle(n, precision, seed=1):
    side = int(np.ceil(n ** (1.0 / 3.0)))
    rng = np.random.default_rng(seed)
    R = 1.9 * np.array([[i % side, i // side % side, i // side ** 2] for i in range(n)], dtype=float)
    R += 0.1 * rng.normal(size=R.shape)
    cfg = kx.sim_config_default(Te=5000.0, precision=precision, kernel=kx.SIM_KERNEL_XL)
    table = kx.param_table(synth.table_to_array(synth.synthetic_table(1)))
    Z = np.ones(n, dtype=np.int32)
    V = synth.maxwell_boltzmann(Z, 300.0, seed=seed)
    return kx.sim_create(cfg, table, Z, R, V=V, charge=n % 2, P0=0.5 * (1.0 - (n % 2) / n) * np.eye(n))


@pytest.mark.parametrize("precision", [kx.SIM_PREC_FP64, kx.SIM_PREC_MIXED])
@pytest.mark.parametrize("n", [1, 2, 3, 5, 33, 63, 64, 65, 100, 127, 128, 129, 160, 161, 255, 256, 257, 320, 321, 384, 385, 481,
                               511, 513, 577, 769, 1023, 1025, 1121, 1730])
def test_eigenpairs_at_the_edges_of_the_launch_shapes(n, precision):
    h = _handle(n, precision)
    try:
        F, Q = kx.sim_get_matrix(h, kx.SIM_MAT_FOCK), kx.sim_get_matrix(h, kx.SIM_MAT_Q)
        eps = kx.sim_get_vector(h, 0)
    finally:
        kx.sim_destroy(h)
    ref = np.linalg.eigvalsh(F)
    width = max(1.0, np.abs(ref).max())
    # eigenvalues: bisection to 1e-12 of the range, tridiagonalisation n 2^-48 (2^-53) |F|
    assert np.abs(eps - ref).max() <= width * (4e-12 + n * 2.0 ** (-46 if precision else -50))
    # vectors: FP64, or the 4-slice products of the back-transformation (2^-24 of sum |a||b|)
    tol = 1e-6 if precision else 1e-10
    assert np.abs(Q.T @ Q - np.eye(n)).max() <= tol
    assert np.abs(F @ Q - Q * eps).max() <= tol * width * 10


@pytest.mark.parametrize("precision", [kx.SIM_PREC_FP64, kx.SIM_PREC_MIXED])
def test_grids_that_do_not_fit_together_give_the_results_of_running_alone(precision):
    """Three threads step an n = 1100 handle each: one grid has a block on every SM, so a
    launch that finds the device taken leaves and its stand-in does the work."""
    def run(seed, out):
        h = _handle(1100, precision, seed)
        try:
            kx.sim_step(h, 6)
            out[seed] = kx.sim_get_state(h, 1100)
        finally:
            kx.sim_destroy(h)

    alone, together = {}, {}
    for seed in (1, 2, 3):
        run(seed, alone)
    threads = [threading.Thread(target=run, args=(s, together)) for s in (1, 2, 3)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for seed in (1, 2, 3):
        for a, b in zip(alone[seed], together[seed]):
            assert np.array_equal(a, b)


@pytest.mark.parametrize("n", [2, 3, 9, 63, 65, 131, 160, 161, 320, 321, 500])
def test_alone_and_beside_others_the_mixed_results_are_the_same(n):
    """Alone: a cluster or a large grid, more lanes an eigenvalue, more threads a pair;
    beside others the small grid.  Same sums in the same order."""
    hs = [_handle(n, kx.SIM_PREC_MIXED, 5) for _ in range(3)]
    try:
        kx.sim_step(hs[0], 3)
        kx.sim_batch_step(hs[1:], 3)
        a, b, c = (kx.sim_get_state(h, n) for h in hs)
    finally:
        for h in hs:
            kx.sim_destroy(h)
    for x, y, z in zip(a, b, c):
        assert np.array_equal(x, y) and np.array_equal(x, z)
