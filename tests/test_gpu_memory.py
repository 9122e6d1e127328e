"""Device memory of a handle."""
import time

import numpy as np
import pytest

import paper_2303_00689_gb300 as kx
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("atoms", [165, 420])
def test_fp64_operands_share_the_eigensolver_workspace(atoms):
    """Mixed handles add 48 n^2 bytes of slices; the digits of an FP64 handle take as much, but lie in
    the workspace of the inverse iteration (5 n^2 doubles)."""
    Z = np.full(atoms, 6, dtype=np.int32)
    n = 4 * atoms
    fp64 = kx.sim_estimate_bytes(kx.sim_config_default(precision=kx.SIM_PREC_FP64), Z)
    mixed = kx.sim_estimate_bytes(kx.sim_config_default(precision=kx.SIM_PREC_MIXED), Z)
    assert fp64 <= mixed - 30 * n * n


@pytest.mark.parametrize("precision", [kx.SIM_PREC_FP64, kx.SIM_PREC_MIXED])
def test_a_served_trajectory_has_no_scratch_for_a_side_stream(precision):
    mol = synth.fullerene_c60(seed=5)
    cfg = kx.sim_config_default(Te=5000.0, precision=precision, scf_max=10, scf_accept=1)
    table = kx.param_table(synth.table_to_array(synth.synthetic_table(1)))
    alone = kx.sim_estimate_bytes(cfg, mol.Z)
    with kx.Server() as srv:
        ticket = srv.submit(cfg, table, mol.Z, mol.R, charge=mol.charge, nsteps=200, records=False)
        used = 0
        while srv.poll(ticket) is None:
            used = max(used, srv.stats()["hbm_in_use"])
            time.sleep(0.002)
    assert 0 < used < alone - 200_000
