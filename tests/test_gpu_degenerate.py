"""Corner weights where corner energies coincide with each other and with grid
energies: bands on a coarse energy lattice, so that most tetrahedra have equal
corners (faces and edges flat, some whole tetrahedra) and every grid energy is
a corner energy of many. The GPU evaluates clamped edge fractions with infinite
reciprocals there; the oracle takes the paper's cases one by one.

Bar: the parity bar of the DOS tests, 2e-5 of the largest value (FP32 weights
of a few roundings each, fixed-point unit below 5e-6 of the maximum)."""
import numpy as np
import pytest

import oracle
from helpers import to_layout

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_orb", [1, 3, 5, 6, 8, 16])
@pytest.mark.parametrize("mode", ["point", "bin", "integrated"])
def test_coinciding_corner_energies(mode, n_orb):
    import paper_1710_10789_gb300 as T

    T.build()
    n = (7, 5, 6)
    rng = np.random.Generator(np.random.PCG64(17))
    nk, nb = n[0] * n[1] * n[2], 4
    eps = np.sort(rng.integers(-4, 5, (nk, nb)) * 0.25, axis=1).astype(np.float32)
    w = rng.uniform(0.0, 1.0, (nk, nb, n_orb)).astype(np.float32)
    omega = (np.arange(-12, 13) * 0.125).astype(np.float32)   # exact in FP32 and FP64
    n_om = len(omega) - (mode == "bin")
    plan = T.Plan(*n, nb, n_orb, n_om, mode=mode)
    E, W = to_layout(eps, w, *n, plan.layout.eps_stride, plan.layout.w_stride)
    out = plan.dos(*(torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (E, W, omega)))
    torch.cuda.synchronize()
    assert plan.status() == T.TETRA_OK
    r = oracle.dos(eps, w, *n, omega.astype(np.float64), mode=mode)
    assert np.max(np.abs(out.cpu().numpy() - r)) <= 2e-5 * np.max(np.abs(r))
