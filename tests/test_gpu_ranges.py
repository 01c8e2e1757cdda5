"""Value ranges and table sizes at which the kernels' counters, units and
shared tables change, against the general path or the oracle."""
import numpy as np
import pytest

import oracle
import tbgen
from helpers import tb_problem, to_layout

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def T():
    import paper_1710_10789_gb300 as T
    T.build()
    return T


@pytest.mark.parametrize("box,bins", [((4, 4, 4), 12900), ((2, 2, 2), 9000)])
def test_batch_flushes_every_block_of_a_long_grid(T, box, bins):
    """A batch whose tile has more blocks of 64 bins than its boxes have work
    items for threads (201 and 141 blocks; 192 and 24 items): one narrow band
    near the top of the grid puts more than 2^31 units into one bin of every
    CTA's 32-bit tile, so the result is right only if that bin's block is
    flushed on the way. The batch equals the single plan bit for bit; the
    band's weight is all in its bin, to the fixed-point unit's 5e-6."""
    n = 64
    top = np.float32(bins * 1e-3 - 0.05)
    edges = (np.arange(bins + 1) * 1e-3).astype(np.float32)
    i = int(np.searchsorted(edges, top, side="right")) - 1
    mid, width = 0.5 * (edges[i] + edges[i + 1]), edges[i + 1] - edges[i]
    noise = np.random.default_rng(3).uniform(-0.3, 0.3, (n ** 3, 1))
    eps = (mid + noise * width).astype(np.float32)
    w = np.full((n ** 3, 1, 1), 0.9, np.float32)
    plan = T.BatchPlan([(n, n, n)], [bins], 1, 1, mode="bin", tune={"box": box})
    E, W = to_layout(eps, w, n, n, n, plan.layouts[0].eps_stride, plan.layouts[0].w_stride)
    Et, Wt, om = torch.from_numpy(E).cuda(), torch.from_numpy(W).cuda(), torch.from_numpy(edges).cuda()
    out, = plan.dos([Et], [Wt], [om])
    assert plan.status() == T.TETRA_OK
    single = T.Plan(n, n, n, 1, 1, bins, mode="bin").dos(Et, Wt, om)
    assert torch.equal(out, single)
    g = out.cpu().numpy()[0].astype(np.float64)
    assert abs(g[i] * float(width) - 0.9) <= 5e-6 * 0.9 and np.count_nonzero(g) == 1


@pytest.mark.parametrize("power", [10, -17])
def test_chi0_real_does_not_depend_on_the_unit_of_energy(T, power):
    """Bands, chemical potential and energies times s (eV as meV: sub-tetrahedra
    hundreds of units wide on a coarse grid; or as 1e5 eV) give Re chi0 / s. s
    is a power of two, so all FP32 products scale exactly and only the
    logarithms round differently: log2 of arguments 2^power larger, rounded at
    |log2| < 32 to 2e-6, in sums that keep 2e-5 of the largest value. The
    oracle at the bar of test_gpu_chi0_real.py, 1e-4."""
    n, q, s = (10, 9, 8), (3, 0, 1), np.float32(2.0 ** power)
    _, eps, _ = tb_problem(3, n)
    mu = float(np.float32(np.median(eps)))
    omega = np.concatenate([tbgen.uniform_grid(-3.0, 3.0, 97), [-25.0, 40.0]]).astype(np.float32)

    def run(s):
        plan = T.Plan(*n, eps.shape[1], 1, 16)
        E, _ = to_layout(eps * s, np.zeros(eps.shape + (1,), np.float32), *n, plan.layout.eps_stride, plan.layout.w_stride)
        r = plan.chi0_real_t0(torch.from_numpy(E).cuda(), q, mu * float(s), torch.from_numpy(omega * s).cuda())
        assert plan.spectral_status() == T.TETRA_OK
        return r.cpu().numpy().astype(np.float64) * float(s)

    one, other = run(np.float32(1)), run(s)
    r = oracle.chi0_real_t0(eps.astype(np.float64), *n, q, mu, omega.astype(np.float64))
    scale = np.max(np.abs(r))
    print(f"2^{power}: {np.max(np.abs(other - one)) / scale:.1e} from 1, {np.max(np.abs(other - r)) / scale:.1e} from the oracle")
    assert np.max(np.abs(other - one)) <= 2e-5 * scale
    assert np.max(np.abs(other - r)) <= 1e-4 * scale


@pytest.mark.parametrize("power", [24, 100])
@pytest.mark.parametrize("n_electrons", [0.37, 5.25])
def test_fermi_level_does_not_depend_on_the_scale_of_the_weights(T, n_electrons, power):
    """Weights and electron count times 2^power: the same level. 2^24 puts the
    count of this grid at 2^66 units of 2^-26 of a tetrahedron. The unit is
    never coarser than 2^-21 of the scaled weight here, 10^5 cells of which
    shift N by 1e-7 of a state at most, and E_F by 1e-6 eV at one state per 10 eV."""
    n = (12, 11, 10)
    _, eps, w = tb_problem(4, n)
    plan = T.Plan(*n, 8, 8, 16)
    E, W = to_layout(eps, w, *n, plan.layout.eps_stride, plan.layout.w_stride)
    Et, Wt = torch.from_numpy(E).cuda(), torch.from_numpy(W).cuda()
    one = plan.fermi_level(Et, Wt, n_electrons)
    s = 2.0 ** power
    assert abs(plan.fermi_level(Et, Wt * s, n_electrons * s) - one) <= 5e-6
    with pytest.raises(T.TetraError) as ex:
        plan.fermi_level(Et, Wt * s, 8.01 * s)
    assert ex.value.status == T.TETRA_EINVAL


@pytest.mark.parametrize("no,bins", [(1, 5600), (3, 2500), (5, 1000), (8, 963), (8, 2000), (16, 600)])
def test_adjoint_tables_too_long_for_shared_memory(T, no, bins):
    """More bins than the adjoint stages in shared memory: its rows in the
    workspace, and without the room for them the values formed at every edge,
    give the same bits."""
    n, nb = (4, 5, 3), 2
    eps, w = (a.astype(np.float32) for a in tbgen.synthetic_bands(29, *n, nb, no))
    edges = tbgen.bin_edges(float(eps.min()) + 0.4, float(eps.max()) - 0.3, bins)
    g = np.random.default_rng(6).normal(0, 1, (no, bins)).astype(np.float32)
    plan = T.Plan(*n, nb, no, bins, mode="bin")
    E, W = to_layout(eps, w, *n, plan.layout.eps_stride, plan.layout.w_stride)
    Et, Wt, om, gt = (torch.from_numpy(a).cuda() for a in (E, W, edges, g))
    ge, gw = plan.dos_backward(Et, Wt, om, gt)
    he, hw = torch.empty_like(ge), torch.empty_like(gw)
    ws = torch.empty(256, dtype=torch.uint8, device="cuda")
    assert T.tetra_dos_backward(plan.handle, Et.data_ptr(), Wt.data_ptr(), om.data_ptr(), gt.data_ptr(), he.data_ptr(),
                                hw.data_ptr(), ws.data_ptr(), 256, torch.cuda.current_stream().cuda_stream) == T.TETRA_OK
    assert torch.equal(ge, he) and torch.equal(gw, hw)


@pytest.mark.parametrize("mode", ["point", "bin", "integrated"])
@pytest.mark.parametrize("no", [1, 3, 8, 16])
def test_large_contributions(T, mode, no, monkeypatch):
    """Contributions beyond the 32-bit tile's bound: weights up to 40 and a
    narrow band, on a coarse energy grid (several copies of the accumulator)
    and on a long one (one). The same bits with a small FLUSH_BITS and other
    boxes, and the oracle within 2e-5 of the largest value."""
    n, nb = (9, 8, 7), 3
    eps, w = (a.astype(np.float32) for a in tbgen.synthetic_bands(41, *n, nb, no))
    w *= 40.0
    eps[:, 0] = eps[:, 0].min() + 1e-3 * (eps[:, 0] - eps[:, 0].min())
    lo, hi = float(eps.min()) - 0.3, float(eps.max()) + 0.3
    for ne in (9, 12000 // (no + 2)):
        om = tbgen.uniform_grid(lo, hi, ne + (mode == "bin"))
        omt = torch.from_numpy(om).cuda()

        def run():
            plan = T.Plan(*n, nb, no, ne, mode=mode)
            E, W = to_layout(eps, w, *n, plan.layout.eps_stride, plan.layout.w_stride)
            out = plan.dos(torch.from_numpy(E).cuda(), torch.from_numpy(W).cuda(), omt)
            assert plan.status() == T.TETRA_OK
            return out

        out = run()
        r = oracle.dos(eps, w, *n, om.astype(np.float64), mode=mode)
        assert np.max(np.abs(out.cpu().numpy() - r)) <= 2e-5 * np.max(np.abs(r))
        for key, value in (("TETRA_FLUSH_BITS", "10"), ("TETRA_BOX_X", "2"), ("TETRA_BOX_Z", "1")):
            monkeypatch.setenv(key, value)
            assert torch.equal(run(), out), key
        for key in ("TETRA_FLUSH_BITS", "TETRA_BOX_X", "TETRA_BOX_Z"):
            monkeypatch.delenv(key)


@pytest.mark.parametrize("mode", ["point", "bin"])
def test_spectral_t0_units_do_not_depend_on_the_length_of_the_grid(T, mode):
    """The unit is 2^-26 of a tetrahedron over the mean spacing, whatever the
    number of energies: a slice of a grid of exact spacing gives the same bits as the
    whole grid does there, down to two energies."""
    n, q = (10, 9, 8), (3, 1, 0)
    _, eps, _ = tb_problem(3, n)
    mu = float(np.median(eps))
    om = torch.arange(-128, 129, device="cuda").float() / 64   # spacing 2^-6
    plan = T.Plan(*n, eps.shape[1], 1, 16)
    E, _ = to_layout(eps, np.zeros(eps.shape + (1,), np.float32), *n, plan.layout.eps_stride, plan.layout.w_stride)
    Et = torch.from_numpy(E).cuda()
    whole = plan.spectral_t0(Et, q, mu, om, mode=mode)
    bins = mode == "bin"
    for a, b in ((0, 256), (20, 90), (100, 117), (160, 162)):
        part = plan.spectral_t0(Et, q, mu, om[a:b + bins].clone(), mode=mode)
        assert plan.spectral_status() == T.TETRA_OK
        assert torch.equal(part, whole[a:b]) and whole[a:b].any(), (a, b)


def test_one_point_has_no_density_of_states(T):
    """A grid of one point: flat bands, a delta that point mode leaves out."""
    plan = T.Plan(1, 1, 1, 2, 3, 5)
    E, W = plan.empty_inputs()
    E[..., :2] = torch.tensor([-0.25, 0.5], device="cuda")
    W += 0.5
    om = torch.tensor([-1.0, -0.25, 0.0, 0.5, 1.0], device="cuda")
    assert not plan.dos(E, W, om).any()


def test_spectral_t0_average_over_one_wide_bin(T):
    """A bin that holds every transition: the average is their total over its
    width, the same factor for all items, so that an error of the quotient does
    not average out. Two roundings of 2^-24 (quotient, result) and 6e-9 for the
    items' own, which do."""
    n, q = (10, 9, 8), (3, 1, 0)
    _, eps, _ = tb_problem(3, n)
    mu, span = float(np.median(eps)), float(eps.max() - eps.min())
    plan = T.Plan(*n, eps.shape[1], 1, 16)
    E, _ = to_layout(eps, np.zeros(eps.shape + (1,), np.float32), *n, plan.layout.eps_stride, plan.layout.w_stride)
    Et = torch.from_numpy(E).cuda()
    total = oracle.spectral_t0(eps.astype(np.float64), *n, q, mu, np.array([0.0, 64.0]), mode="bin")[0] * 64.0
    widths = (span + np.random.default_rng(8).uniform(0.1, 20.0, 64)).astype(np.float32)
    worst = 0.0
    for width in widths:
        om = torch.tensor([0.0, float(width)], device="cuda")
        g = float(plan.spectral_t0(Et, q, mu, om, mode="bin")[0])
        worst = max(worst, abs(g * float(width) / total - 1.0))
    print(f"{worst:.2e}")
    assert worst <= 2.0 ** -23 + 6e-9
