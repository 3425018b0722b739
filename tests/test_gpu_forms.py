"""Kernels that a rule or the tuner chooses between, each form made to run:
resident model steps with every cluster size, the grouped triangular sweeps
with 4 and 8 particles per CTA on a factor whose widest steps exceed the ring
of entries in shared memory, and the solves of a layout too large for them."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1910_01031_gb300 import iewpf, synth
from gpu_common import ensemble, oracle_problem, start_state

pytestmark = pytest.mark.gpu


# the cluster sizes that hold the grid: slabs of at least 4 rows and at most 200 KB
@pytest.mark.parametrize("nx,ny,c,fits", [(16, 17, 1, (2, 4)), (33, 35, 1, (2, 4, 8)), (64, 64, 3, (2, 4, 8)),
                                          (50, 49, 3, (2, 4, 8)), (96, 45, 3, (2, 4, 8)), (128, 64, 3, (4, 8)),
                                          (160, 160, 3, ())])
def test_every_cluster_size_equals_the_march(nx, ny, c, fits):
    """Forecasts with and without model error and with a fixed number of scheme steps, bit for bit, with the
    same counters; the resident form shown by its launches: one per model step in place of the scheme steps'."""
    cfg = synth.Config("edge", nx, ny, n_particles=3, c_omega=c)
    U32, _ = start_state(cfg, 3)

    def run(ens):
        ens.set_state(U32)
        n0, w0 = ens.launch_count(), ens.work()
        ens.forecast_fixed(2, False, 14)
        n1 = ens.launch_count()
        ens.forecast(2, True)
        ens.forecast(1, False)
        return ens.get_state(), tuple(ens.last_nsub()), ens.work() - w0, ens.counters(), n1 - n0

    march = ensemble(cfg)
    march.set_stepper(1, 2, 16, 4)
    assert march.resident() == 0
    want = run(march)
    for ctas in (2, 4, 8):
        ens = ensemble(cfg)
        if ctas not in fits:
            with pytest.raises(iewpf.IewpfError):
                ens.set_resident(ctas)
            continue
        ens.set_resident(ctas)
        got = run(ens)
        assert ens.resident() == ctas
        assert np.array_equal(got[0], want[0]), ctas
        assert got[1:4] == want[1:4], ctas
        assert want[4] - got[4] >= 2 * 14, (got[4], want[4])
        ens.set_resident(0)
        assert run(ens)[4] == want[4]
    with pytest.raises(iewpf.IewpfError):
        march.set_resident(3)


# 20 groups of 8 x 8 moorings on neighbouring cells, each coupled throughout, and one of 8 x 16: columns 104 to 126
# of the groups' factors make steps of 20 rows and more than 2048 entries, the long group's go on after them
@pytest.mark.parametrize("ne,particles_per_cta", [(1, 4), (13, 4), (613, 8)])
def test_grouped_sweeps_over_steps_larger_than_the_ring(ne, particles_per_cta):
    """Against the batch's sweeps, a warp per particle, bit for bit."""
    import torch
    cells = np.array([(4 + 48 * (k % 5) + i, 4 + 40 * (k // 5) + j) for k in range(20) for j in range(8) for i in range(8)] +
                     [(250 + i, 4 + j) for j in range(16) for i in range(8)])
    n_obs = len(cells)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert iewpf.solve_group(2 * n_obs, ne, sms) == particles_per_cta
    cfg = synth.Config("edge", 280, 160, n_particles=ne, n_obs=n_obs, obs_kind=synth.OBS_MOORING, c_omega=1)
    xy = synth.cell_positions(cfg, cells)
    batch = iewpf.Batch([iewpf.params_from_config(cfg)], [xy])
    single = ensemble(cfg, mooring_xy=xy)
    # the groups' factors are dense: 128 * 127 / 2 entries each, and more in the long one
    assert single.factor_info()[1] > 20 * 128 * 127 // 2
    U = np.repeat(synth.initial_state(cfg, min(ne, 20), seed=7).astype(np.float32), -(-ne // 20), axis=0)[:ne]
    y = synth.obs_from_state(cfg, synth.initial_particle(cfg, 77, seed=5), cells, synth.obs_noise(cfg, n_obs, 0))
    for e in (single, batch.instances[0]):
        e.set_state(U)
    diag = batch.cycle(2, [(None, y)])
    single.forecast(1, True)
    single.forecast(1, False)
    d = single.assimilate(None, y)
    assert diag[0, 0] == d["w_target"] and diag[0, 1] == d["beta"] and diag[0, 2] == 0
    assert np.array_equal(batch.instances[0].get_state(), single.get_state())


def test_layouts_larger_than_any_group():
    """3136 moorings apart from each other (6272 unknowns: too many for a group of 4, and for a warp's vector in
    shared memory): phi of every particle against the 2 x 2 blocks solved one by one in FP64, 1e-9."""
    m, spacing, ne = 56, 16, 3
    n = m * spacing + 16
    cfg = synth.Config("edge", n, n, n_particles=ne, n_obs=m * m, obs_kind=synth.OBS_MOORING, c_omega=1)
    assert iewpf.solve_group(2 * m * m, ne) == 1
    cells = np.array([[8 + spacing * (k % m), 8 + spacing * (k // m)] for k in range(m * m)])
    P = oracle_problem(cfg)
    ens = ensemble(cfg, mooring_xy=synth.cell_positions(cfg, cells))
    U32, U64 = start_state(cfg, ne)
    y = synth.obs_from_state(cfg, synth.initial_particle(cfg, 77, seed=5), cells, synth.obs_noise(cfg, m * m, 0))
    ens.set_state(U32)
    d = ens.assimilate(None, y)
    block = O.hqht(P, O.pull_stencil(P), [tuple(cells[0])]) + cfg.obs_sigma ** 2 * np.eye(2)
    inn = np.asarray(O.innovations(P, U64, [tuple(c) for c in cells], y)).reshape(ne, m * m, 2)
    ref = np.einsum("pli,ij,plj->p", inn, np.linalg.inv(block), inn)
    np.testing.assert_allclose(d["phi"], ref, rtol=1e-9)
