"""Kernel variants at the sizes where their dispatch or their tiling changes, against the FP64 oracle
(tolerances of the other parity tests: FP64 forces 1e-11 of rms(F), energies 1e-12)."""
import numpy as np
import pytest

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
