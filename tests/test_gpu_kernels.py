"""Kernel variants at the sizes where their dispatch or their tiling changes, against the FP64 oracle
(tolerances of the other parity tests: FP64 forces 1e-11 of rms(F), energies 1e-12)."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_1012_2677_gb300 import ljmd, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("list_form", [ljmd.LJ_LIST_FULL, ljmd.LJ_LIST_HALF])
@pytest.mark.parametrize("M,rho,rc,margin", [
    (6, 0.5, 2.5, 0.5),    # 3 cells per side, one cell per tile: fewer keys than a warp's turn
    (10, 0.9, 3.5, 1.0),   # 147 keys per tile (more than one turn of the warps), rows longer than
                           # a warp's queue, segments beyond shared memory
    (11, 0.9, 4.5, 1.0),   # 5,324 staged particles: beyond the FP64 kernel's tile, the general kernel
])
def test_fp64_tiles(M, rho, rc, margin, list_form):
    p = O.LJParams(rc_over_sigma=rc)
    x, L = O.fcc_lattice(M, rho)
    x = synth.dyadic(O.wrap(x + synth.displacements(len(x), 0.06, 3), L))
    F, pe, vir = O.forces(x, L, p)
    with ljmd.System(cutoff=rc, margin=margin, precision=ljmd.LJ_FP64, list_form=list_form) as s:
        s.set_state(x, None, L)
        s.compute_forces()
        _, _, gf, _ = s.get_state()
        gpe, _, gvir = s.energies()
    rms = np.sqrt((F ** 2).sum(1).mean())
    assert np.sqrt(((gf - F) ** 2).sum(1)).max() / rms <= 1e-11
    assert gpe == pytest.approx(pe, rel=1e-12) and gvir == pytest.approx(vir, rel=1e-12)


@pytest.mark.parametrize("precision,tol", [(ljmd.LJ_MIXED, 2e-4), (ljmd.LJ_FP64, 1e-10)])
@pytest.mark.parametrize("M,rho,rc,margin", [
    (5, 1.0, 2.5, 0.6),    # fewer than three cells per side: no tiles
    (6, 0.5, 2.5, 0.5),    # 3 cells per side: fewer keys than a warp's turn
    (10, 0.9, 3.5, 1.0),   # long rows, segments beyond shared memory
    (11, 0.9, 4.5, 1.0),   # beyond the FP64 queue kernel's tile
])
def test_adjoint_tiles(M, rho, rc, margin, precision, tol):
    """Tolerances of the other tests of the Hessian-vector product and the parameter derivatives."""
    p = O.LJParams(rc_over_sigma=rc)
    x, L = O.fcc_lattice(M, rho)
    x = synth.dyadic(O.wrap(x + synth.displacements(len(x), 0.06, 3), L))
    w = synth.gaussian((len(x), 3), 11)
    ref = O.hvp(x, L, w, p)
    dpe, vjp = O.param_derivs(x, L, p, lam=w)
    with ljmd.System(cutoff=rc, margin=margin, precision=precision) as s:
        s.set_state(x, None, L)
        hw, dth = s.hvp(w)
    rms = np.sqrt((ref ** 2).sum(1).mean())
    assert np.sqrt(((hw - ref) ** 2).sum(1)).max() / rms <= tol
    for got, want in zip(dth, (vjp[0], vjp[1], dpe[0], dpe[1])):
        assert got == pytest.approx(want, rel=max(tol, 1e-12), abs=tol * 1e-3 * abs(dpe[0]))


@pytest.mark.parametrize("precision,list_form", [(ljmd.LJ_MIXED, ljmd.LJ_LIST_FULL), (ljmd.LJ_MIXED, ljmd.LJ_LIST_HALF),
                                                 (ljmd.LJ_FP64, ljmd.LJ_LIST_FULL), (ljmd.LJ_FP64, ljmd.LJ_LIST_HALF)])
@pytest.mark.parametrize("M,rho,every,mode,steps", [
    (5, 0.4, 1, ljmd.LJ_VALID_HALF_MARGIN, (7, 33)),   # 3 cells per side; a second call continues the first
    (8, 0.6, 3, ljmd.LJ_VALID_HALF_MARGIN, (40,)),     # energies every third step
    (9, 0.9, 0, ljmd.LJ_VALID_DUTC, (1, 39)),          # dense, the DUTC rule, no energies; a single step
    (6, 0.5, 1, ljmd.LJ_VALID_HALF_MARGIN, (300,)),    # more steps than one run takes
])
def test_resident_run_matches_separate_launches(M, rho, every, mode, steps, precision, list_form):
    """A box whose tiles fit on the chip takes its steps in one launch; with the phase timers on, the same
    steps are separate launches.  Positions agree to the drift that one rounding of every force makes in 40
    steps (dt^2 40^2 / 2 times 1e-5 of rms(F) < 50 in the mixed form, 1e-11 in the FP64 form), the energy
    logs have the same records; after 300 steps the energies agree to the drift test's scale."""
    out = []
    for timed in (False, True):
        log = torch.zeros((400, 4), dtype=torch.float64, device="cuda")
        with ljmd.System(cutoff=2.5, margin=0.4, precision=precision, list_form=list_form, energy_every=every) as s:
            s.init_lattice(M, rho, 1.1, 7)
            s.set_validity(mode)
            s.set_energy_log(log)
            s.set_profiling(timed)
            for k in steps:
                s.step(0.004, k)
            x, v, _, img = s.get_state()
            st = s.stats()
            out.append((x + img * s.box, v, st, log.cpu().numpy(), s.energies()))
    (xa, va, sa, la, ea), (xb, vb, sb, lb, eb) = out
    assert sa["steps"] == sb["steps"] == sum(steps) and sa["status_word"] == sb["status_word"] == 0
    assert sa["kernel_launches"] < sb["kernel_launches"]
    assert np.array_equal(la[:, 0], lb[:, 0])
    n = np.count_nonzero(lb[:, 1])
    if sum(steps) <= 40:
        tol = 8e-6 if precision == ljmd.LJ_MIXED else 8e-12
        assert np.abs(xa - xb).max() <= tol
        assert sa["rebuilds"] == sb["rebuilds"]
        etol = 1e-6 if precision == ljmd.LJ_MIXED else 1e-11
        assert np.allclose(la[:n, 1:], lb[:n, 1:], rtol=etol, atol=etol * np.abs(lb[:n, 1:]).max() if n else 0)
    else:
        tot = lambda l: l[:n, 1] + l[:n, 2]  # noqa: E731
        assert np.abs(tot(la) - tot(lb)).max() <= 1e-3 * np.abs(lb[:n, 1]).max()
    assert ea[0] == pytest.approx(eb[0], rel=1e-2 if sum(steps) > 40 else 1e-5)


@pytest.mark.parametrize("precision", [ljmd.LJ_MIXED, ljmd.LJ_FP64])
@pytest.mark.parametrize("n,cells,spread", [
    (1, 3, 1.0), (255, 4, 1.0), (256, 4, 1.0), (257, 4, 1.0),  # blocks of 256 particles
    (2500, 6, 0.3),   # most cells empty, counts far beyond what the mean suggests
    (3000, 18, 1.0), (3000, 19, 1.0),   # the last box that one launch reorders, the first that it does not
])
def test_reordering_of_small_boxes(n, cells, spread, precision):
    """Cell starts, cell order (ids ascending) and pairs are integers: they equal the oracle's."""
    L = cells * 3.05
    x = synth.dyadic(np.random.default_rng(n + cells).uniform(0.0, spread * L, (n, 3)))
    x[::7] += L  # outside the box: folded
    v = synth.gaussian(x.shape, 9)
    with ljmd.System(cutoff=2.5, margin=0.5, precision=precision) as s:
        s.set_state(x, v, L)
        for _ in range(2):  # the second construction starts from the first one's order
            s.build_pairlist()
            assert s.stats()["cells_per_side"] == cells
            ptr, lst = s.grid()
            xw = x - np.floor(x / L) * L
            c = np.minimum((xw * (cells / L)).astype(np.int64), cells - 1)
            cell = (c[:, 0] * cells + c[:, 1]) * cells + c[:, 2]
            order = np.lexsort((np.arange(n), cell))
            assert np.array_equal(ptr[:cells ** 3], np.searchsorted(cell[order], np.arange(cells ** 3)))
            assert np.array_equal(lst, order)
            assert np.array_equal(s.pairs(), O.pairs_within(xw, L, 3.0))
        xs, vs, _, img = s.get_state()
        assert np.array_equal(xs + img * L, x) and np.array_equal(vs, v)


@pytest.mark.parametrize("precision,list_form", [(ljmd.LJ_MIXED, ljmd.LJ_LIST_FULL), (ljmd.LJ_FP64, ljmd.LJ_LIST_FULL)])
def test_overlapping_launches_match_separate_ones(precision, list_form):
    """The launches of a run of steps may start while the one before them ends; with the phase timers on, none
    does.  The same kernels: the same bits, also where the list expires inside a run."""
    x, L = O.fcc_lattice(44, 0.5)
    x = x[:-1]  # 340,735 particles: more than a resident run takes
    v = synth.gaussian(x.shape, 5)
    out = []
    for timed in (False, True):
        log = torch.zeros((64, 4), dtype=torch.float64, device="cuda")
        with ljmd.System(cutoff=2.5, margin=0.4, precision=precision, list_form=list_form, energy_every=3) as s:
            s.set_state(x, v, L)
            s.set_energy_log(log)
            s.set_profiling(timed)
            for k in (1, 23, 6):
                s.step(0.004, k)
            st = s.stats()
            assert st["status_word"] == 0 and st["rebuilds"] >= 3
            out.append((*s.get_state(), log.cpu().numpy()[:, 0], st["rebuilds"], st["kernel_launches"]))
    assert out[0][-1] >= 60 and out[0][-2:] == out[1][-2:]
    for a, b in zip(out[0][:-2], out[1][:-2]):
        assert np.array_equal(a, b)
