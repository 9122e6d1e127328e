"""Eigenpairs of the Fock matrix where the kernels of the eigensolver exchange data: the same
matrix gives the same bits every time, at the sizes where the exchange can go wrong."""
import os
import subprocess
import sys
import threading

import numpy as np
import pytest

import paper_2303_00689_gb300 as kx
import synth

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def lattice(n, precision, seed=1, **cfg):
    """A lattice of n H atoms (one orbital each)."""
    side = int(np.ceil(n ** (1.0 / 3.0)))
    rng = np.random.default_rng(seed)
    R = 1.9 * np.array([[i % side, i // side % side, i // side ** 2] for i in range(n)], dtype=float)
    R += 0.1 * rng.normal(size=R.shape)
    cfg = kx.sim_config_default(Te=5000.0, precision=precision, **{"kernel": kx.SIM_KERNEL_XL, **cfg})
    table = kx.param_table(synth.table_to_array(synth.synthetic_table(1)))
    Z = np.ones(n, dtype=np.int32)
    V = synth.maxwell_boltzmann(Z, 300.0, seed=seed)
    return kx.sim_create(cfg, table, Z, R, V=V, charge=n % 2, P0=0.5 * (1.0 - (n % 2) / n) * np.eye(n))


def eigenpairs(h):
    return kx.sim_get_vector(h, 0), kx.sim_get_matrix(h, kx.SIM_MAT_Q)


@pytest.mark.parametrize("n", [2, 3, 17, 26, 33, 48, 63, 64])
def test_one_block_gives_the_same_bits_every_time(n):
    """Four groups of threads hand each other a column's products through shared memory."""
    h = lattice(n, kx.SIM_PREC_FP64)
    try:
        eps, Q = eigenpairs(h)
        ref = np.linalg.eigvalsh(kx.sim_get_matrix(h, kx.SIM_MAT_FOCK))
        assert np.abs(eps - ref).max() <= max(1.0, np.abs(ref).max()) * (4e-12 + n * 2.0 ** -50)
        for _ in range(40):
            kx.sim_set_state(h)
            e, q = eigenpairs(h)
            assert np.array_equal(e, eps) and np.array_equal(q, Q)
    finally:
        kx.sim_destroy(h)


@pytest.mark.parametrize("n", [70, 128, 131, 300])
def test_a_limit_that_may_expire_in_any_column_leaves_the_handle_usable(n):
    """With a limit of 1 ns a poll gives up as soon as it looks at the clock, so a step may end in
    any column: every warp of every block leaves, and the same state then gives the same bits."""
    h = lattice(n, kx.SIM_PREC_FP64)
    try:
        ref = eigenpairs(h)
        for _ in range(10):
            kx.sim_debug_barrier_limit(1)
            try:
                kx.sim_set_state(h)
            except kx.SimError as e:
                assert e.code == kx.SIM_ETIMEOUT
            finally:
                kx.sim_debug_barrier_limit(2_000_000_000)
        kx.sim_set_state(h)
        for a, b in zip(ref, eigenpairs(h)):
            assert np.array_equal(a, b)
    finally:
        kx.sim_destroy(h)


def residuals(n, precision):
    """Largest entries of Q^T Q - I and of F Q - Q eps over the spectral range."""
    h = lattice(n, precision)
    try:
        eps, Q = eigenpairs(h)
        F = kx.sim_get_matrix(h, kx.SIM_MAT_FOCK)
    finally:
        kx.sim_destroy(h)
    return np.abs(Q.T @ Q - np.eye(n)).max(), np.abs(F @ Q - Q * eps).max() / max(1.0, np.abs(eps).max())


@pytest.mark.parametrize("n", [1997, 1998, 2002, 2003])
def test_grids_at_the_shared_memory_limit_of_a_plain_launch(n):
    """Dynamic and static shared memory of the small (1997, 1998) or the large grid are just above
    48 KB: a launch without the opt-in is refused, so in a process that has launched nothing larger."""
    code = ("import sys; sys.path.insert(0, '.'); import paper_2303_00689_gb300 as kx\n"
            "from tests.test_gpu_eigen import residuals\n"
            f"print(*residuals({n}, kx.SIM_PREC_MIXED))")
    out = subprocess.run([sys.executable, "-c", code], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert out.returncode == 0, out.stderr
    # 4-slice products of the back-transformation: 2^-24 of sum |a||b|
    orthogonality, residual = map(float, out.stdout.split())
    assert orthogonality <= 1e-6 and residual <= 1e-5


def test_the_largest_mixed_size_that_fits_shared_memory():
    """n = 9255 (2313 C, 3 H): three vectors of the double-float grid fill an SM's shared memory."""
    Z = np.array([6] * 2313 + [1] * 3, dtype=np.int32)
    n, side = 9255, 14
    R = 2.6 * np.array([[i % side, i // side % side, i // side ** 2] for i in range(len(Z))], dtype=float)
    R += 0.1 * np.random.default_rng(1).normal(size=R.shape)
    cfg = kx.sim_config_default(Te=5000.0, precision=kx.SIM_PREC_MIXED, kernel=kx.SIM_KERNEL_XL, m_max=1, m_min=1)
    table = kx.param_table(synth.table_to_array(synth.synthetic_table(1)))
    h = kx.sim_create(cfg, table, Z, R, charge=1, P0=4627.0 / n * np.eye(n))
    try:
        eps, Q = eigenpairs(h)
        F = kx.sim_get_matrix(h, kx.SIM_MAT_FOCK)
    finally:
        kx.sim_destroy(h)
    some = np.linspace(0, n - 1, 40).astype(int)
    assert np.abs(F @ Q[:, some] - Q[:, some] * eps[some]).max() <= 1e-5 * max(1.0, np.abs(eps).max())
    assert np.abs(Q.T @ Q[:, some] - np.eye(n)[:, some]).max() <= 1e-6


@pytest.mark.parametrize("precision", [kx.SIM_PREC_FP64, kx.SIM_PREC_MIXED])
@pytest.mark.parametrize("n", [1, 2, 9, 64, 65, 131, 300, 608, 609, 900, 1217])
def test_alone_and_beside_others_the_results_are_the_same(n, precision):
    """Grids, lanes per eigenvalue and threads per pair differ beside other handles, results do not:
    stepped alone, by sim_batch_step (launches, and the handles' graphs), in one graph of a batch."""
    hs = [lattice(n, precision, 5, kernel=kx.SIM_KERNEL_KRYLOV, m_max=2, m_min=2) for _ in range(7)]
    batch = None
    try:
        for h in hs[3:5]:
            kx.sim_enable_graphs(h)
        kx.sim_step(hs[0], 2)
        kx.sim_batch_step(hs[1:3], 2)
        kx.sim_batch_step(hs[3:5], 2)
        batch = kx.sim_batch_create(hs[5:])
        kx.sim_batch_run(batch, 2)
        ref = [*kx.sim_get_state(hs[0], n), *eigenpairs(hs[0])]
        for h in hs[1:]:
            for a, b in zip(ref, [*kx.sim_get_state(h, n), *eigenpairs(h)]):
                assert np.array_equal(a, b)
    finally:
        if batch:
            kx.sim_batch_destroy(batch)
        for h in hs:
            kx.sim_destroy(h)


@pytest.mark.parametrize("n", [1801, 2050, 2401, 2561, 3361])
def test_fp64_with_rows_outside_shared_memory(n):
    """Several launches with a hand-over between them, rows in L2 beside resident ones (n = 2050 and
    above), and the shapes of the largest systems."""
    h = lattice(n, kx.SIM_PREC_FP64, m_max=1, m_min=1)
    try:
        eps, Q = eigenpairs(h)
        F = kx.sim_get_matrix(h, kx.SIM_MAT_FOCK)
    finally:
        kx.sim_destroy(h)
    some = np.linspace(0, n - 1, 60).astype(int)
    width = max(1.0, np.abs(eps).max())
    assert np.abs(np.linalg.eigvalsh(F) - eps).max() <= width * (4e-12 + n * 2.0 ** -50)
    assert np.abs(F @ Q[:, some] - Q[:, some] * eps[some]).max() <= 1e-9 * width
    assert np.abs(Q.T @ Q[:, some] - np.eye(n)[:, some]).max() <= 1e-10


@pytest.mark.parametrize("n,count", [(1000, 2), (2050, 3)])
def test_fp64_small_grids_and_large_grids_that_meet(n, count):
    """Beside others the small grid, with rows in L2; three threads at n = 2050 (four launches a
    tridiagonalisation) so that a launch behind others may leave the work to its stand-in."""
    hs = [lattice(n, kx.SIM_PREC_FP64, 1, m_max=1, m_min=1) for _ in range(count + 1)]
    try:
        kx.sim_step(hs[0], 3)
        ref = [*kx.sim_get_state(hs[0], n), *eigenpairs(hs[0])]
        if count == 2:
            kx.sim_batch_step(hs[1:], 3)
        else:
            ts = [threading.Thread(target=kx.sim_step, args=(h, 3)) for h in hs[1:]]
            for t in ts:
                t.start()
            for t in ts:
                t.join()
        for h in hs[1:]:
            for a, b in zip(ref, [*kx.sim_get_state(h, n), *eigenpairs(h)]):
                assert np.array_equal(a, b)
    finally:
        for h in hs:
            kx.sim_destroy(h)


@pytest.mark.parametrize("precision", [kx.SIM_PREC_FP64, kx.SIM_PREC_MIXED])
def test_a_served_trajectory_has_the_bits_of_running_alone(precision):
    """n = 240: in the server no cluster, a small grid, fewer lanes per eigenvalue, no side stream."""
    mol = synth.fullerene_c60(seed=5)
    cfg = kx.sim_config_default(Te=5000.0, precision=precision, scf_max=10, scf_accept=1, m_max=2, m_min=2)
    table = kx.param_table(synth.table_to_array(synth.synthetic_table(1)))
    with kx.Server() as srv:
        tickets = [srv.submit(cfg, table, mol.Z, mol.R, charge=mol.charge, nsteps=4) for _ in range(3)]
        srv.drain(120.0)
        served = [srv.poll(t) for t in tickets]
    h = kx.sim_create(cfg, table, mol.Z, mol.R, charge=mol.charge)
    try:
        records = kx.sim_step(h, 4)
        R, V, F, _ = kx.sim_get_state(h, mol.natoms)
    finally:
        kx.sim_destroy(h)
    for s in served:
        assert s["status"] == kx.SIM_OK and s["records"] == records
        assert np.array_equal(s["R"], R) and np.array_equal(s["V"], V) and np.array_equal(s["F"], F)
