"""GPU kernels at the sizes where their work splits can go wrong (edges of
tiles and slices, remainders, smallest and largest of a rule's range),
against the FP64 oracle; tolerances as in the parity tests of each quantity."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1910_01031_gb300 import iewpf, synth
from gpu_common import ensemble, oracle_problem, rel_l2, start_state

pytestmark = pytest.mark.gpu


def _observed(cfg, n, cycle=0):
    """Drifter positions, their cells and observed values from another draw of the initial state."""
    xy = synth.drifter_positions(cfg, n)
    cells = [O.obs_cell(oracle_problem(cfg), *p) for p in xy]
    truth = synth.initial_state(cfg, 1, seed=3)[0]
    return xy, cells, synth.obs_from_state(cfg, truth, np.array(cells), synth.obs_noise(cfg, n, cycle))


@pytest.mark.parametrize("ne", [31, 33, 4097])
@pytest.mark.parametrize("scheme", [iewpf.TWO_STAGE, iewpf.ONE_STAGE])
def test_ensemble_wide_step_over_slices(ne, scheme):
    """The ensemble-wide step runs in slices of 32 particles (64 above 4096): target, beta, alpha and
    weights of every particle against the oracle's on the same c, gamma, zeta (1e-10, as iewpf_weights)."""
    cfg = synth.Config("edge_48x48", 48, 48, n_particles=ne, n_obs=2)
    ens = iewpf.Ensemble(iewpf.params_from_config(cfg, scheme=scheme))
    U = np.repeat(synth.initial_state(cfg, min(ne, 40), seed=7).astype(np.float32), -(-ne // 40), axis=0)[:ne]
    ens.set_state(U)
    xy, _, y = _observed(cfg, 2)
    d = ens.assimilate(xy, y)
    N = 3.0 * cfg.nx * cfg.ny
    ref = O.iewpf_scalars_one_stage(d["c"], d["gamma"], N) if scheme == iewpf.ONE_STAGE else \
        O.iewpf_scalars(d["c"], d["gamma"], d["zeta"], N)
    np.testing.assert_allclose(d["w_target"], ref.get("w_target", ref["cbar"]), rtol=1e-10)
    np.testing.assert_allclose(d["cbar"], ref["cbar"], rtol=1e-10)
    np.testing.assert_allclose(d["beta"], ref["beta"], rtol=1e-10, atol=1e-300)
    np.testing.assert_allclose(d["alpha"], ref["alpha"], rtol=1e-10)
    np.testing.assert_allclose(d["neglogw"], ref["neglogw"], rtol=1e-10)


@pytest.mark.parametrize("nx,ny", [(48, 48), (51, 48), (51, 51), (51, 57), (54, 57), (150, 141), (384, 375)])
def test_random_vectors_over_philox_blocks(nx, ny):
    """Coarse grids of every remainder modulo 4 (the last Philox block partly used) and of one and several
    slices of the dot products: gamma and zeta at 1e-10, the state (which carries the projection of nu~
    and the posterior field) at 1e-5."""
    cfg = synth.Config("edge", nx, ny, n_particles=3, n_obs=1)
    ens, P = ensemble(cfg), oracle_problem(cfg)
    U32, U64 = start_state(cfg, 3)
    ens.set_state(U32)
    xy, cells, y = _observed(cfg, 1)
    d = ens.assimilate(xy, y)
    ref, dref = O.assimilate(P, U64, cells, y, t=0)
    np.testing.assert_allclose(d["gamma"], dref["gamma"], rtol=1e-10)
    np.testing.assert_allclose(d["zeta"], dref["zeta"], rtol=1e-10)
    assert rel_l2(ens.get_state(), ref) <= 1e-5



# particles per CTA of the fine stage: 1, 4 and 16 (the largest groups the ensemble fills the GPU with)
@pytest.mark.parametrize("ne", [3, 305, 1233])
@pytest.mark.parametrize("nx,ny,c", [(48, 50, 3), (65, 47, 1), (97, 75, 5)])
def test_fine_stage_groups_and_tile_edges(nx, ny, c, ne):
    """Analysis update and Q^{1/2} on grids that do not fill their 64 x 32 tiles and 32-column strips, with
    observations whose stencils wrap both seams, for every particle grouping; sampled particles (first,
    last, group edges) against the oracle at 1e-5."""
    cfg = synth.Config("edge", nx, ny, n_particles=ne, n_obs=3, c_omega=c)
    ens, P = ensemble(cfg), oracle_problem(cfg)
    base = synth.initial_state(cfg, 7, seed=7).astype(np.float32)
    U32 = base[np.arange(ne) % 7]
    ens.set_state(U32)
    xy = np.array([[0.2 * cfg.dx, 0.4 * cfg.dy], [(nx - 0.5) * cfg.dx, 0.5 * ny * cfg.dy], [33.5 * cfg.dx, 32.5 * cfg.dy]])
    cells = [O.obs_cell(P, *p) for p in xy]
    y = synth.obs_from_state(cfg, synth.initial_state(cfg, 1, seed=3)[0], np.array(cells), synth.obs_noise(cfg, 3, 0))
    d = ens.assimilate(xy, y)
    got = ens.get_state()
    sample = sorted({0, ne - 1, min(ne - 1, 3), min(ne - 1, 4), min(ne - 1, 15), min(ne - 1, 16), ne // 2})
    for i in sample:
        ref, _ = O.assimilate(P, U32[i:i + 1].astype(np.float64), cells, y, t=0, p0=i,
                              scalars={"beta": d["beta"], "alpha": d["alpha"][i:i + 1]})
        assert rel_l2(got[i], ref[0]) <= 1e-5
    x = np.random.default_rng(3).standard_normal((ne, P.N_R)).astype(np.float32)
    ens.set_state(U32)
    ens.add_qhalf(x)
    got = ens.get_state()
    for i in sample:
        assert rel_l2(got[i], O.add_qhalf(P, x[i].astype(np.float64), U32[i].astype(np.float64))) <= 1e-5


@pytest.mark.parametrize("nx,ny", [(44, 46), (64, 64), (66, 47), (96, 45), (93, 50), (97, 44), (176, 48)])
def test_marching_shapes_agree_bitwise_and_with_the_oracle(nx, ny):
    """Rows that close on a ring of lanes (44, 64, 96, 93 with 3 columns, 66) or take strips with halo (one
    and several, with and without remainder), chunks from 2 rows to more than the grid: every kind and
    shape gives the same bits, and the oracle's state at 1e-5."""
    cfg = synth.Config("edge", nx, ny, n_particles=3)
    ens, P = ensemble(cfg), oracle_problem(cfg)
    U32, U64 = start_state(cfg, 3)
    first = None
    for kind in (1, 2):
        for nc in (2, 3, 4):
            for rows, warps in ((2, 4), (ny // 3, 2), (ny, 8), (2 * ny, 1)):
                ens.set_stepper(kind, nc, rows, warps)
                ens.set_state(U32)
                ens.set_counters(0, 0)
                ens.forecast(1, False)
                got = ens.get_state()
                if first is None:
                    first = got
                    ref, _, _ = O.forecast(P, U64, 1, False, t0=0)
                    assert rel_l2(got, ref) <= 1e-5
                assert np.array_equal(got, first), (kind, nc, rows, warps)


@pytest.mark.parametrize("nx,ny,c", [(16, 17, 1), (33, 35, 1), (64, 64, 3), (50, 49, 3), (96, 45, 3), (128, 64, 3)])
def test_resident_model_steps_equal_the_march(nx, ny, c):
    """Grids small enough to stay in a cluster's shared memory (uneven slabs, rows of one to four blocks of
    32 columns, more rows than warps): tuned forecasts, with and without model error and with a fixed number
    of scheme steps, against the marched ones bit for bit, with the same counters of work and scheme steps."""
    cfg = synth.Config("edge", nx, ny, n_particles=3, c_omega=c)
    U32, _ = start_state(cfg, 3)
    a, b = ensemble(cfg), ensemble(cfg)
    shape = a.tune()
    b.set_stepper(*shape)
    for e in (a, b):
        e.set_state(U32)
    w0 = a.work()
    for e in (a, b):
        e.forecast(2, True)
        e.forecast(1, False)
        e.forecast_fixed(1, True, 14)
    assert np.array_equal(a.get_state(), b.get_state())
    assert np.array_equal(a.last_nsub(), b.last_nsub())
    assert a.work() - w0 == b.work()
    assert a.counters() == b.counters()


@pytest.mark.parametrize("m,spacing,ne", [(16, 5, 1), (17, 5, 9), (17, 8, 6), (36, 5, 611)])
def test_grouped_sweeps_equal_a_warp_per_particle(m, spacing, ne):
    """Layouts of 256 moorings and more: the triangular sweeps of 4 or 8 particles per CTA (ragged last groups,
    coupled and uncoupled factors) against the batch's, which take a warp per particle, bit for bit."""
    n = 16 * (-(-(m * spacing + 8) // 16))
    cfg = synth.Config("edge", n, n, n_particles=ne, n_obs=m * m, obs_kind=synth.OBS_MOORING, c_omega=1)
    cells = np.array([[4 + spacing * (k % m), 3 + spacing * (k // m)] for k in range(m * m)])
    xy = synth.cell_positions(cfg, cells)
    batch = iewpf.Batch([iewpf.params_from_config(cfg)], [xy])
    single = ensemble(cfg, mooring_xy=xy)
    U = np.repeat(synth.initial_state(cfg, min(ne, 20), seed=7).astype(np.float32), -(-ne // 20), axis=0)[:ne]
    y = synth.obs_from_state(cfg, synth.initial_particle(cfg, 77, seed=5), cells, synth.obs_noise(cfg, m * m, 0))
    for e in (single, batch.instances[0]):
        e.set_state(U)
    diag = batch.cycle(2, [(None, y)])
    single.forecast(1, True)
    single.forecast(1, False)
    d = single.assimilate(None, y)
    assert diag[0, 0] == d["w_target"] and diag[0, 1] == d["beta"] and diag[0, 2] == 0
    assert np.array_equal(batch.instances[0].get_state(), single.get_state())


@pytest.mark.parametrize("positions", ["same", "overlapping", "wrapping", "apart"])
@pytest.mark.parametrize("n", [1, 2, 3, 13])
def test_local_blocks_in_sequence(n, positions):
    """Local blocks applied one after another (inputs loaded two blocks ahead, the two blocks before patched
    in): fewer blocks than the look-ahead, blocks on one place, sharing points with one or both predecessors,
    over the periodic edges and apart, against the oracle's products in FP64 at 1e-5 of the state."""
    cfg = synth.Config("edge", 96, 93, n_particles=3, n_obs=n)
    ens, P = ensemble(cfg), oracle_problem(cfg)
    U32, U64 = start_state(cfg, 3)
    ens.set_state(U32)
    step = {"same": (0, 0), "overlapping": (7, 4), "wrapping": (40, 88), "apart": (29, 24)}[positions]
    cells = np.array([[(5 + step[0] * k) % 96, (3 + step[1] * k) % 93] for k in range(n)])
    xy = synth.cell_positions(cfg, cells)
    y = synth.obs_from_state(cfg, synth.initial_particle(cfg, 77, seed=5), cells, synth.obs_noise(cfg, n, 0))
    ens.assimilate(xy, y)
    ref, _ = O.assimilate(P, U64, [tuple(c) for c in cells], y, t=0)
    assert rel_l2(ens.get_state(), ref) <= 1e-5


@pytest.mark.parametrize("n,spread", [(15, 40), (16, 40), (33, 40), (64, 40), (79, 40), (40, 12), (64, 3), (80, 40)])
def test_factor_by_levels_equals_column_by_column(n, spread):
    """Drifter layouts whose factor is made level by level (32 to 159 unknowns that mostly do not interact) or
    column by column (fewer, more, or clustered), against the batch's, which goes column by column, bit for bit."""
    cfg = synth.Config("edge", 352, 336, n_particles=2, n_obs=n, c_omega=1)
    rng = np.random.default_rng(n + spread)
    cells = np.array([[(spread * (k % 8) + rng.integers(0, 9)) % 352, (spread * (k // 8) + rng.integers(0, 9)) % 336]
                      for k in range(n)])
    xy = synth.cell_positions(cfg, cells)
    batch, single = iewpf.Batch([iewpf.params_from_config(cfg)], None), ensemble(cfg)
    U = synth.initial_state(cfg, 2, seed=7).astype(np.float32)
    y = synth.obs_from_state(cfg, synth.initial_particle(cfg, 77, seed=5), cells, synth.obs_noise(cfg, n, 0))
    for e in (single, batch.instances[0]):
        e.set_state(U)
    diag = batch.cycle(2, [(xy, y)])
    single.forecast(1, True)
    single.forecast(1, False)
    d = single.assimilate(xy, y)
    assert diag[0, 0] == d["w_target"] and diag[0, 1] == d["beta"] and diag[0, 2] == 0
    assert np.array_equal(batch.instances[0].get_state(), single.get_state())


@pytest.mark.parametrize("nx,ny,offset", [(64, 64, 0), (64, 64, 1), (64, 64, 4), (45, 47, 0), (50, 46, 2), (150, 141, 3)])
def test_device_state_copies(nx, ny, offset):
    """States in and out of device memory by 16 bytes or by single values (planes of any remainder, arrays off
    their alignment), particles in either buffer: the copies through host memory, bit for bit."""
    import torch
    cfg = synth.Config("edge", nx, ny, n_particles=5)
    U32, _ = start_state(cfg, 5)
    U32[3] *= np.float32(1.5)                # other wave speeds: other numbers of scheme steps
    a, b = ensemble(cfg), ensemble(cfg)
    flat = torch.zeros(offset + U32.size + 8, dtype=torch.float32, device="cuda")
    view = flat[offset:offset + U32.size].view(*U32.shape)
    view.copy_(torch.from_numpy(U32))
    a.set_state(view)
    b.set_state(U32)
    for steps in (0, 1, 1):
        if steps:
            a.forecast(steps, True)
            b.forecast(steps, True)
        flat.fill_(-1.0)
        a.get_state(view)
        assert np.array_equal(view.cpu().numpy(), b.get_state())
        assert bool((flat[:offset] == -1).all()) and bool((flat[offset + U32.size:] == -1).all())


@pytest.mark.parametrize("nx,ny,c", [(16, 16, 1), (17, 18, 1), (36, 37, 1), (37, 67, 1), (68, 39, 1), (48, 54, 3), (107, 51, 3)])
def test_coarse_correlation_over_row_groups(nx, ny, c):
    """The 5 x 5 SOAR sums in groups of four rows with the periodic seam apart: coarse grids of one column of
    blocks and more, every remainder of rows, one model step with model error against the oracle at 1e-5."""
    cfg = synth.Config("edge", nx, ny, n_particles=3, c_omega=c)
    ens, P = ensemble(cfg), oracle_problem(cfg)
    U32, U64 = start_state(cfg, 3)
    ens.set_state(U32)
    ens.forecast(1, True)
    ref, _, _ = O.forecast(P, U64, 1, True, t0=0)
    assert rel_l2(ens.get_state(), ref) <= 1e-5
