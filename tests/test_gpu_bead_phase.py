"""Bead phase at the places where its FP32 arithmetic or its lists could go wrong,
against FP64 references: neighbours across a periodic edge, slow beads,
supports that span a periodic box, fibers that have drifted far, supports about
as large as a list.
"""
import math
import os

import numpy as np
import pytest

import oracle
from paper_2212_14153_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

THREADS = min(16, os.cpu_count() or 1)


@pytest.fixture(scope="module")
def fpd():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2212_14153_gb300 import build, fpd as binding
    build.build()
    return binding


def box(nx, ny, a, xi, centres, n_beads, force, precision, **kw):
    """Beads pushed through fluid at rest in a doubly periodic box."""
    nb = n_beads * len(centres)
    cfg = dict(nx=nx, ny=ny, u_bottom=0.0, u_top=0.0, nu_f=1.0 / 6.0, re=1.0, visc_ratio=50.0, xi=xi, a=a,
               n_beads=n_beads, n_fibers=len(centres), k_s=-1.0, k_b=0.0, stiffness_K=0.0, k_ev=-1.0, phi_cut=8.0,
               collision=0, s_e=1.64, s_eps=1.54, s_q=1.9, init_couette=0, periodic_y=1, bead_fx=force[0],
               bead_fy=force[1], gx=-force[0] * nb / (nx * ny), gy=-force[1] * nb / (nx * ny), centres=centres,
               theta0=[0.0] * len(centres), precision=precision)
    cfg.update(kw)
    return cfg


@pytest.mark.parametrize("axis", [0, 1])
def test_neighbours_across_the_edge_of_a_wide_lattice_vs_oracle(fpd, axis):
    # a fiber over the periodic edge of 65536 columns (or 65535 rows), whose FP32
    # positions have an ulp of 2^-8: the offset between beads on either side
    # must not be rounded there.  An offset of up to 16 cells rounded to FP32
    # (4.8e-7) twice, at a slope of phi of 1 / (2 xi) = 1 / 3, and phi's own
    # 1.5e-7 make an error below 5e-7 a neighbour, of which there are four; V is
    # a mean of these.  The beads on the right lie 0.45 of an ulp of the left
    # ones' positions off that grid.
    n = (65536, 64) if axis == 0 else (64, 65535)
    at = 2.0 + 0.45 / 256.0
    centre = [at, 32.2] if axis == 0 else [32.2, at]
    cfg = box(*n, 2.0, 1.5, [centre], 5, (1e-3, 7e-4), 1, theta0=[axis * math.pi / 2])
    sim, ref = fpd.Simulation(cfg), oracle.Sim(dict(cfg, precision=0, threads=THREADS))
    sim.step(2)  # one bead phase: the force density is a third of V
    ref.step(2)
    V, rV = sim.beads()[1], ref.beads()[1]
    sim.close()
    e = np.abs(V - rV).max() / np.abs(rV).max()
    print(f"axis {axis}: V {e:.1e}")
    assert e < 1e-5


@pytest.mark.parametrize("force", [1e-4, 1e-8, 1e-12, 1e-18])
def test_slow_beads_keep_their_relative_accuracy(fpd, force):
    # the flow a weak force drives is linear in it: the FP32 path keeps the
    # relative accuracy it has at ordinary speeds (FP32 arithmetic over 20
    # steps: below 1e-5, as against the oracle) down to any speed
    cfg = box(48, 40, 2.0, 0.5, [[47.2, 12.7]], 1, (force, -0.6 * force), 1)
    V = []
    for precision in (0, 1):
        sim = fpd.Simulation(dict(cfg, precision=precision))
        sim.step(20)
        V.append(sim.beads()[1][0])
        sim.close()
    e = np.abs(V[1] - V[0]).max() / np.abs(V[0]).max()
    print(f"force {force:.0e}: V {np.abs(V[0]).max():.1e}, error {e:.1e}")
    assert e < 1e-5


@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("centre", [[10.0, 10.2], [19.9, 0.4], [3.5, 14.8]])
def test_support_that_spans_a_periodic_box(fpd, precision, centre):
    # S = sum phi over the nearest images where phi is still 5e-3 half a box
    # away, of a bead carried along by a uniform flow.  400 values of phi with
    # errors of at most 4e-7 against S = 114 in FP32
    L, a, xi = 20, 6.0, 1.5
    # the wall speeds only set FP16's scale here: y is periodic
    cfg = box(L, L, a, xi, [centre], 1, (0.0, 0.0), precision, visc_ratio=1.0, u_bottom=-0.2, u_top=0.2)
    sim = fpd.Simulation(cfg)
    f = oracle.feq(1.0, 0.31, -0.17)[:, None, None]
    sim.set_populations(np.ascontiguousarray(np.broadcast_to(f, (9, L, L))))
    c = np.arange(L) + 0.5
    for n in range(6):
        R, V, _, S = sim.beads()
        assert n < 2 or abs(V[0, 0]) > 0.1
        d = [x - L * np.floor(x / L + 0.5) for x in (c - R[0, 0], c - R[0, 1])]
        r = np.hypot(d[0][None, :], d[1][:, None])
        want = np.where(r < a + 8.0 * xi, 0.5 * (np.tanh((a - r) / xi) + 1.0), 0.0).sum()
        print(f"precision {precision}, step {n}: S {S[0]:.6f}, error {abs(S[0] / want - 1):.1e}")
        assert abs(S[0] / want - 1) < (1e-13 if precision == 0 else 2e-6)
        sim.step(1)
    sim.close()


@pytest.mark.parametrize("n_beads", [6, 20])  # forces in a cluster; by the last CTA
@pytest.mark.parametrize("periods", [0, 4096, 16384])
def test_forces_do_not_depend_on_how_far_a_fiber_has_drifted(fpd, n_beads, periods):
    # stiff springs stretched by up to 1e-4 after any number of passes over the
    # periodic edge: the FP32 paths' force against the FP64 one at the same
    # positions.  Roundings of FP32 (6e-8 each): the stretch from a difference of
    # squares, a product with the tangent and a sum of two pulls, six or so.
    rng = np.random.default_rng(n_beads)
    nx, l0 = 128, 4.0
    d = l0 + rng.uniform(-1e-4, 1e-4, n_beads)
    t = 0.3 + 0.02 * np.arange(n_beads)
    xy = np.stack([20.0 + np.cumsum(d * np.cos(t)), 8.0 + np.cumsum(d * np.sin(t))], 1)
    xy = np.round(xy * 2.0 ** 24) / 2.0 ** 24  # exact after the shift as well
    xy[:, 0] += periods * nx
    cfg = box(nx, 128, 2.0, 0.5, [[0.0, 0.0]], n_beads, (0.0, 0.0), 1, bead_xy=xy, k_ev=0.0)
    sim = fpd.Simulation(cfg)
    k_s = 0.25 * math.pi * 4.0 * l0 ** 2
    for steps in (0, 3):
        sim.step(steps)
        R, _, F, _ = sim.beads()
        want = oracle.bead_forces(R, n_beads, 1, 2.0, k_s, 0.0, 0.0)
        e = np.abs(F - want).max() / np.abs(want).max()
        print(f"{n_beads} beads, {periods} periods, {steps} steps: F {e:.1e}")
        assert e < 1e-6
    sim.close()


@pytest.mark.parametrize("precision,xi", [
    (1, 1.4375), (1, 1.5), (2, 1.4375), (2, 1.5),  # boxes of 35 x 35 and 36 x 36, lists of 1280
    (0, 1.1875), (0, 1.25),                        # 31 x 31 and 32 x 32, lists of 1000
])
def test_support_boxes_about_as_large_as_a_list(fpd, precision, xi):
    # more beads than SMs run in the narrowest CTAs, each with all of its
    # bead's cells; alone an instance's CTAs are wide or share a bead.  The same
    # bits, on either side of a list's length
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    rng = np.random.default_rng(7)
    n = sms // 16 + 2
    cases = [wl.random_fiber(rng, 150, 90, n_beads=8, a=4.0, xi=xi, n_fibers=2, precision=precision, theta0=[0.4, 2.5])
             for _ in range(n)]
    b = fpd.Batch(precision, n, 512 << 20, 16 * n)
    slots = [b.add(c, 6) for c in cases]
    while b.run(100):
        pass
    for c, s in list(zip(cases, slots))[::3]:
        alone = fpd.Simulation(c)
        alone.step(6)
        assert np.array_equal(alone.populations(), b.populations(s))
        for x, y in zip(alone.beads(), b.beads(s)):
            assert np.array_equal(x, y)
        alone.close()
    if precision != 2:
        ref = oracle.Sim(dict(cases[0], precision=0, threads=THREADS))
        ref.step(6)
        for x, y in zip(b.beads(slots[0])[:2], ref.beads()[:2]):
            assert np.linalg.norm(x - y) < (1e-12 if precision == 0 else 2e-5) * np.linalg.norm(y)
    b.close()


@pytest.mark.parametrize("xi", [1.4375, 1.5])
def test_support_box_of_two_lists_beside_a_long_sweep(fpd, xi):
    # 4290 tiles: the bead CTAs wait for the sweep first, with 256 threads and
    # lists of 1280 cells (FP32 against the oracle)
    rng = np.random.default_rng(9)
    cfg = wl.random_fiber(rng, 1030, 1040, n_beads=9, a=4.0, xi=xi, n_fibers=2, precision=1)
    sim, ref = fpd.Simulation(cfg), oracle.Sim(dict(cfg, precision=0, threads=THREADS))
    sim.step(10)
    ref.step(10)
    for x, y in zip(sim.beads()[:2], ref.beads()[:2]):
        assert np.linalg.norm(x - y) < 2e-5 * np.linalg.norm(y)
    sim.close()


@pytest.mark.parametrize("precision", [1, 2])
@pytest.mark.parametrize("xi", [0.875, 0.9375, 1.0])  # boxes of 484, 529 and 576 cells
def test_widths_of_the_bead_ctas_give_the_same_bits(fpd, precision, xi):
    # 18 beads: 256 threads with a box of up to 512 cells, 512 above; in a
    # batch of 11 such instances 128
    rng = np.random.default_rng(5)
    cases = [wl.random_fiber(rng, 180, 70, n_beads=9, a=2.25, xi=xi, n_fibers=2, precision=precision) for _ in range(11)]
    b = fpd.Batch(precision, 11, 256 << 20, 198)
    slots = [b.add(c, 8) for c in cases]
    while b.run(100):
        pass
    for c, s in list(zip(cases, slots))[::5]:
        alone = fpd.Simulation(c)
        alone.step(8)
        assert np.array_equal(alone.populations(), b.populations(s))
        for x, y in zip(alone.beads(), b.beads(s)):
            assert np.array_equal(x, y)
        alone.close()
    b.close()
