"""Calls at the limits of the kernels' capacities, units and waits: what was built for an ordinary liquid
must stay right, be refused cleanly or give up cleanly outside it."""
import numpy as np
import pytest

import oracle as O
from paper_1012_2677_gb300 import ljmd, synth

pytestmark = pytest.mark.gpu


def _min_image(d, L):
    return d - L * np.round(d / L)


def test_batch_tile_beyond_the_capacities_is_skipped_alone():
    """The capacities of a batch are fixed at the host construction.  Replica 0 contracts (v = -1.6 (x - centre), an
    FCC gas of rho 0.2: its density triples in 60 steps and no pair comes close), so a later device-side
    construction makes tiles beyond 1.4 times the largest there was: the call must end with LJ_EDEVICE and the
    status bit, and every other replica, whose tiles go through the same buffers after the skipped ones (98 tiles
    a replica, 608 buffers on the chip), must be where a single system takes it: 60 steps accumulate at most
    dt^2 60^2 / 2 times the force difference of the two summation orders (1e-5 of |F| < 10), 3e-6, and less than
    ten times that with the growth of a difference over 0.24 time units."""
    R, N, rho, dt, steps = 20, 2000, 0.2, 0.004, 60
    xs, vs = [], []
    for r in range(R):
        x, L = synth.fcc_thinned(N, rho, 40 + r)
        xs.append(synth.dyadic(x))
        vs.append(synth.dyadic(-1.6 * (xs[0] - 0.5 * L) if r == 0 else synth.thermal_velocities(N, 1.0, 60 + r)))
    x, v = np.concatenate(xs), np.concatenate(vs)
    bx, bv, bf = (np.empty_like(x) for _ in range(3))
    with ljmd.Batch([N] * R, [L] * R, cutoff=2.5, margin=0.3) as b:
        assert b.stats()["tiles"] > 152 * 4 + 98
        b.set_state(x, v)
        with pytest.raises(ljmd.LjmdError) as e:
            b.step(dt, steps)
        assert e.value.code == ljmd.LJ_EDEVICE
        assert b.stats()["status_word"] & (ljmd.LJ_ST_CELL_RANGE | ljmd.LJ_ST_LIST_OVERFLOW)
        assert not b.stats()["status_word"] & (ljmd.LJ_ST_TIMEOUT | ljmd.LJ_ST_NONFINITE)
        with pytest.raises(ljmd.LjmdError):  # the arrays are filled; the status is still raised
            ljmd._chk(ljmd.load().ljmd_batch_get_state(b.h, *(a.ctypes.data for a in (bx, bv, bf)), 0), "get_state")
    for r in range(1, R):
        with ljmd.System(cutoff=2.5, margin=0.3, precision=ljmd.LJ_MIXED) as s:
            s.set_state(xs[r], vs[r], L)
            s.step(dt, steps)
            sx, _, _, _ = s.get_state()
        assert np.abs(_min_image(bx[r * N:(r + 1) * N] - sx, L)).max() < 3e-5, r


def _liquid(N, rho, seed):
    x, L = synth.fcc_thinned(N, rho, seed)
    return O.wrap(x + synth.displacements(N, 0.05, seed + 1), L), L


def _droplet(N, L, seed):
    """A ball of N particles at density 0.95 in a box that is otherwise empty."""
    x, l = _liquid(8 * N // 4, 0.95, seed)
    r = np.sqrt(((x - 0.5 * l) ** 2).sum(1))
    return x[np.argsort(r)[:N]] - 0.5 * l + 0.5 * L, L


@pytest.mark.parametrize("rc,make", [
    (3.5, lambda: [_liquid(6000, 0.8, 3), _liquid(900, 0.5, 4)]),
    (4.5, lambda: [_liquid(9000, 0.85, 5), _liquid(2500, 0.4, 6)]),
    (5.0, lambda: [_droplet(10000, 66.0, 7), _liquid(2500, 0.5, 8)]),  # tiles by the mean count do not fit here
])
def test_batch_with_a_long_cutoff(rc, make):
    """Cells of a long search length hold many particles: the default tiles must still fit."""
    boxes = make()
    xs = [synth.dyadic(x) for x, _ in boxes]
    n, box = [len(x) for x in xs], [L for _, L in boxes]
    x = np.concatenate(xs)
    v = synth.dyadic(synth.thermal_velocities(len(x), 0.7, 9))
    with ljmd.Batch(n, box, cutoff=rc, margin=0.5) as b:
        b.set_state(x, v)
        pe, _, _ = b.energies()
        b.set_state(x, v)
        _, _, f = b.get_state()
        b.step(0.002, 11, graph_steps=5)
        bx, _, _ = b.get_state()
        assert b.stats()["status_word"] == 0
    o = 0
    for r, xr in enumerate(xs):
        sl = slice(o, o + n[r])
        F, pe_o, _ = O.forces(xr, box[r], O.LJParams(rc_over_sigma=rc))
        assert np.sqrt(((f[sl] - F) ** 2).sum(1)).max() / np.sqrt((F ** 2).sum(1).mean()) <= 1e-5
        assert pe[r] == pytest.approx(pe_o, rel=1e-6)
        with ljmd.System(cutoff=rc, margin=0.5, precision=ljmd.LJ_MIXED) as s:
            s.set_state(xr, v[sl], box[r])
            s.step(0.002, 11)
            sx, _, _, _ = s.get_state()
        assert np.abs(_min_image(bx[sl] - sx, box[r])).max() < 1e-5
        o += n[r]


TINY = 16  # SM clock cycles: no wait of a kernel is over that fast


def _state_whatever_the_status(s, n):
    x, v, f = (np.empty((n, 3)) for _ in range(3))
    img = np.empty((n, 3), dtype=np.int32)
    ljmd.load().ljmd_get_state(s.h, *(a.ctypes.data for a in (x, v, f, img)), 0)
    return x, v, f, img


# 10,700 particles in 27 cells: the tile capacities guessed from the mean counts do not fit in shared memory (237 KB
# of 227), the ones measured afterwards do (221 KB)
@pytest.mark.parametrize("N,rho,rc,guess_fits", [(4000, 0.5, 2.5, True), (10700, 0.94, 6.9, False)])
def test_reordering_of_a_small_box_times_out(N, rho, rc, guess_fits):
    x, L = synth.fcc_thinned(N, rho, 5)
    x = synth.dyadic(O.wrap(x + synth.displacements(N, 0.03, 6), L))
    v = synth.dyadic(synth.thermal_velocities(N, 1.0, 7))
    with ljmd.System(cutoff=rc, margin=0.5, precision=ljmd.LJ_MIXED, list_form=ljmd.LJ_LIST_FULL) as s:
        s.set_state(x, v, L)
        ljmd.ljmd_set_wait_budget(TINY)
        try:
            with pytest.raises(ljmd.LjmdError) as e:
                s.build_pairlist()
        finally:
            ljmd.ljmd_set_wait_budget(0)
        assert e.value.code == ljmd.LJ_EDEVICE
        st = s.stats()
        assert st["status_word"] == ljmd.LJ_ST_TIMEOUT and st["rebuilds"] == 0
        if not guess_fits:  # given up before the list kernel: the reordering is the only launch
            assert st["kernel_launches"] == 1
        gx, gv, _, img = _state_whatever_the_status(s, N)
        assert np.array_equal(gx, x) and np.array_equal(gv, v) and not img.any()
    with ljmd.System(cutoff=rc, margin=0.5, precision=ljmd.LJ_MIXED, list_form=ljmd.LJ_LIST_FULL) as s:
        s.set_state(x, v, L)
        s.compute_forces()
        _, _, f, _ = s.get_state()
    F, _, _ = O.forces(x, L, O.LJParams(rc_over_sigma=rc))
    assert np.sqrt(((f - F) ** 2).sum(1)).max() / np.sqrt((F ** 2).sum(1).mean()) <= 1e-5


@pytest.mark.parametrize("list_form", [ljmd.LJ_LIST_FULL, ljmd.LJ_LIST_HALF])
@pytest.mark.parametrize("sigma", [50.0, 1e-3, 1e-5, 3.4e-10])
def test_fp64_form_in_any_unit_of_length(sigma, list_form):
    """The FP64 form's results do not depend on the unit of length (argon in metres: sigma = 3.4e-10): forces,
    energies and the Hessian-vector product with the tolerances of the other FP64 tests, and a few steps of a box
    that runs resident.  Positions and box are multiples of the storage's last bit q (2^-50 beside the offset 4 of
    a small box; 2^-42 at least where the box is 715), so that nothing is rounded on the way in.  A step rounds a
    stored position by q / 2 at most, and the image of a particle outside the box by as much; through the forces
    (K dt^2 < 0.01) that adds a hundredth: five steps stay within 4 q of the oracle's."""
    q = 2.0 ** (-50 if sigma < 1.0 else -41)
    p = O.LJParams(sigma=sigma, rc_over_sigma=2.5)
    x, L = O.fcc_lattice(8, 0.7)
    x = O.wrap(x + synth.displacements(len(x), 0.06, 3), L)
    x, L = np.round(x * sigma / q) * q, np.round(L * sigma / q) * q
    w = synth.gaussian(x.shape, 11)
    F, pe, vir = O.forces(x, L, p)
    with ljmd.System(sigma=sigma, cutoff=2.5 * sigma, margin=0.5 * sigma, precision=ljmd.LJ_FP64,
                     list_form=list_form) as s:
        s.set_state(x, w, L)
        s.compute_forces()
        _, _, f, _ = s.get_state()
        gpe, _, gvir = s.energies()
        assert np.sqrt(((f - F) ** 2).sum(1)).max() / np.sqrt((F ** 2).sum(1).mean()) <= 1e-11
        assert gpe == pytest.approx(pe, rel=1e-12) and gvir == pytest.approx(vir, rel=1e-12)
        s.step(0.002 * sigma, 5)
        xs, _, _, img = s.get_state()
        xo, *_ = O.vv_run(x, w, L, 0.002 * sigma, 5, p)
        assert np.abs(xs + img * L - xo).max() <= 4 * q
    if list_form == ljmd.LJ_LIST_FULL:
        ref = O.hvp(x, L, w, p)
        with ljmd.System(sigma=sigma, cutoff=2.5 * sigma, margin=0.5 * sigma, precision=ljmd.LJ_FP64) as s:
            s.set_state(x, None, L)
            hw, _ = s.hvp(w)
        assert np.sqrt(((hw - ref) ** 2).sum(1)).max() / np.sqrt((ref ** 2).sum(1).mean()) <= 1e-10


def test_batch_autotuner_knows_the_default():
    """A batch whose force launch takes 164 us with the tiles of tile_cells = 6 and 130 us with the default's: the
    autotuner, which keeps the fastest, must not leave it slower than it found it."""
    x, L = synth.fcc_thinned(20000, 0.3, 5)
    x = O.wrap(x + synth.displacements(len(x), 0.05, 6), L)
    with ljmd.Batch([len(x)] * 40, [L] * 40, cutoff=2.5, margin=0.3) as b:
        b.set_state(np.tile(x, (40, 1)))
        default = b.time_force(20)
        tile, lanes, _ = b.autotune(trials=10)
        assert tile == b.stats()["tile_cells"] == 10
        assert b.time_force(20) <= 1.1 * default


def test_dilute_fp64_box_holds_no_staging_descriptors():
    """256 cells per side, 4.2 million tiles: 8 bytes a tile for its list segment (34 MB) beside three words a cell
    (201 MB).  The 192 bytes a tile that only the mixed form's pipelined kernel reads would add 805 MB."""
    torch = pytest.importorskip("torch")
    x = synth.uniform_positions(1000, 769.0, 3)
    with ljmd.System(cutoff=2.5, margin=0.5, precision=ljmd.LJ_FP64) as s:
        s.set_state(x, None, 769.0)
        torch.cuda.synchronize()
        free0, _ = torch.cuda.mem_get_info()
        s.build_pairlist()
        free1, _ = torch.cuda.mem_get_info()
        assert s.stats()["cells_per_side"] == 256
        assert free0 - free1 < 300e6
        assert np.array_equal(s.pairs(), O.pairs_within(x, 769.0, 3.0))


def test_a_refused_list_leaves_no_list_behind():
    """A cutoff whose cells are beyond what a tile can stage (16,384 particles in 27 cells) is refused; the
    particles are in the new cells' order by then, so the former list is gone: forces are refused too until a
    list can be built again."""
    x, L = O.fcc_lattice(16, 1.0)
    x = synth.dyadic(O.wrap(x + synth.displacements(len(x), 0.03, 6), L))
    with ljmd.System(cutoff=2.5, margin=0.5, precision=ljmd.LJ_MIXED) as s:
        s.set_state(x, None, L)
        s.compute_forces()
        for call in (lambda: s.build_pairlist(7.5, 0.5), s.compute_forces, lambda: s.step(0.001, 1)):
            with pytest.raises(ljmd.LjmdError) as e:
                call()
            assert e.value.code == ljmd.LJ_ERANGE
        s.build_pairlist(2.5, 0.5)
        s.compute_forces()
        gx, _, f, _ = s.get_state()
        assert np.array_equal(gx, x) and s.stats()["status_word"] == 0
    F, _, _ = O.forces(x, L)
    assert np.sqrt(((f - F) ** 2).sum(1)).max() / np.sqrt((F ** 2).sum(1).mean()) <= 1e-5


def test_fp64_tiles_around_the_queue_kernels_capacity():
    """27 cells, each tile stages the whole box: from about 4,520 particles on the queue kernel's tile does not fit
    beside its static shared memory, and the general kernel takes over without a gap."""
    for N in range(4492, 4557, 4):
        x, L = _liquid(N, 0.9, 11)
        with ljmd.System(cutoff=5.0, margin=0.5, precision=ljmd.LJ_FP64, list_form=ljmd.LJ_LIST_FULL) as s:
            s.set_state(synth.dyadic(x), None, L)
            s.compute_forces()
            assert s.stats()["cells_per_side"] == 3
            _, _, f, _ = s.get_state()
        F, _, _ = O.forces(synth.dyadic(x), L, O.LJParams(rc_over_sigma=5.0))
        assert np.sqrt(((f - F) ** 2).sum(1)).max() / np.sqrt((F ** 2).sum(1).mean()) <= 1e-11, N


def test_first_step_of_a_resident_box_allocates_nothing():
    """Beyond the list construction, which comes before: 32,000 particles, no energies asked for."""
    torch = pytest.importorskip("torch")
    with ljmd.System(cutoff=2.5, margin=0.5, precision=ljmd.LJ_MIXED, list_form=ljmd.LJ_LIST_FULL, energy_every=0) as s:
        s.init_lattice(20, 0.5, 1.0, 1)
        s.build_pairlist()
        torch.cuda.synchronize()
        free0, _ = torch.cuda.mem_get_info()
        n0 = s.stats()["kernel_launches"]
        s.step(0.001, 3)
        free1, _ = torch.cuda.mem_get_info()
        assert s.stats()["kernel_launches"] - n0 == 1  # one resident run
        assert free1 == free0


def _gives_up(s, call):
    """call with the short budget ends with LJ_EDEVICE or, where it does not look at the status itself, leaves it."""
    ljmd.ljmd_set_wait_budget(TINY)
    try:
        try:
            call()
        except ljmd.LjmdError as e:
            assert e.code == ljmd.LJ_EDEVICE
    finally:
        ljmd.ljmd_set_wait_budget(0)
    assert s.stats()["status_word"] == ljmd.LJ_ST_TIMEOUT


def _device_still_usable():
    x, L = _liquid(2000, 0.6, 5)
    x = synth.dyadic(x)
    F, _, _ = O.forces(x, L)
    with ljmd.System(cutoff=2.5, margin=0.5, precision=ljmd.LJ_FP64) as s:
        s.set_state(x, None, L)
        s.step(0.0, 1)
        _, _, f, _ = s.get_state()
        assert s.stats()["status_word"] == 0
    assert np.sqrt(((f - F) ** 2).sum(1)).max() / np.sqrt((F ** 2).sum(1).mean()) <= 1e-11


@pytest.mark.parametrize("list_form", [ljmd.LJ_LIST_FULL, ljmd.LJ_LIST_HALF])
def test_list_kernel_wait_times_out(list_form):
    """8,000 cells: more than the one-launch reordering takes, so nothing gives up before the list kernel."""
    with ljmd.System(cutoff=2.5, margin=0.5, precision=ljmd.LJ_MIXED, list_form=list_form) as s:
        s.init_lattice(30, 0.5, 1.0, 1)
        _gives_up(s, s.build_pairlist)
        assert s.stats()["cells_per_side"] == 20 and s.stats()["kernel_launches"] > 2
    _device_still_usable()


@pytest.mark.parametrize("list_form", [ljmd.LJ_LIST_FULL, ljmd.LJ_LIST_HALF])
@pytest.mark.parametrize("precision", [ljmd.LJ_MIXED, ljmd.LJ_FP64])
def test_grid_barrier_of_a_resident_run_times_out(precision, list_form):
    with ljmd.System(cutoff=2.5, margin=0.5, precision=precision, list_form=list_form, energy_every=1) as s:
        s.init_lattice(10, 0.5, 1.0, 1)
        s.build_pairlist()
        n0 = s.stats()["kernel_launches"]
        _gives_up(s, lambda: s.step(0.005, 5))
        assert s.stats()["kernel_launches"] - n0 == 1
        with pytest.raises(ljmd.LjmdError):  # the run's state is not to be had
            s.step(0.005, 1)
    _device_still_usable()


def test_waits_of_the_fp64_queue_kernels_time_out():
    with ljmd.System(cutoff=2.5, margin=0.5, precision=ljmd.LJ_FP64) as s:
        s.init_lattice(20, 0.5, 1.0, 1)
        s.build_pairlist()
        _gives_up(s, s.compute_forces)
    with ljmd.System(cutoff=2.5, margin=0.5, precision=ljmd.LJ_FP64, list_form=ljmd.LJ_LIST_FULL) as s:
        s.init_lattice(10, 0.5, 1.0, 1)
        s.build_pairlist()
        _gives_up(s, lambda: s.hvp(np.ones((4000, 3))))
    _device_still_usable()
