"""Kernels at the edges of their tiles and dispatch rules, against the oracle:
grids of one point to just beyond a tile, every orbital-count instantiation,
few items per box (lanes share a walk), tables too large for shared memory,
unaligned outputs, unsorted energies, contributions too large for the 32-bit
tiles.

Bounds: DOS and occupation 2e-5 of the largest value (the parity bar; the
fixed-point unit keeps the rounding below 5e-6 of it); gradients as in
test_gpu_grad.py (1e-5 and 1e-4 of the largest entry); the susceptibility 1e-4
(real part) and 2e-5 of the largest value; Fermi levels 1e-4 eV (FP32
energies)."""
import numpy as np
import pytest

import oracle
import tbgen
from helpers import from_layout, to_layout

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def T():
    import paper_1710_10789_gb300 as T
    T.build()
    return T


def bands(seed, n, nb, no):
    eps, w = tbgen.synthetic_bands(seed, *n, nb, no)
    return eps.astype(np.float32), w.astype(np.float32)


def tensors(plan, eps, w, n, dtype=None):
    E, W = to_layout(eps, w, *n, plan.layout.eps_stride, plan.layout.w_stride)
    Et, Wt = torch.from_numpy(E).cuda(), torch.from_numpy(W).cuda()
    return Et, Wt if dtype is None else Wt.to(dtype)


def close(g, r, tol):
    scale = np.max(np.abs(r))
    assert scale > 0 and np.max(np.abs(g - r)) <= tol * scale, np.max(np.abs(g - r)) / scale


@pytest.mark.parametrize("mode", ["point", "bin", "integrated"])
@pytest.mark.parametrize("n,nb,no,nw", [((1, 1, 1), 1, 1, 5), ((2, 3, 1), 1, 1, 40), ((9, 17, 5), 1, 1, 700),
                                        ((8, 9, 7), 2, 3, 300), ((11, 5, 6), 3, 5, 200), ((7, 10, 3), 6, 6, 90),
                                        ((16, 16, 4), 7, 7, 150), ((33, 3, 9), 8, 8, 400)])
def test_dos_shapes(T, n, nb, no, nw, mode, monkeypatch):
    eps, w = bands(11, n, nb, no)
    lo, hi = float(eps.min()) - 0.3, float(eps.max()) + 0.3
    om = tbgen.uniform_grid(lo, hi, nw + (mode == "bin"))
    plan = T.Plan(*n, nb, no, nw, mode=mode)
    Et, Wt = tensors(plan, eps, w, n)
    omt = torch.from_numpy(om).cuda()
    g = plan.dos(Et, Wt, omt)
    torch.cuda.synchronize()
    assert plan.status() == T.TETRA_OK
    r = oracle.dos(eps, w, *n, om.astype(np.float64), mode=mode)
    if np.max(np.abs(r)) > 0:   # (one point: flat bands, a delta in point mode)
        close(g.cpu().numpy(), r, 2e-5)
    # another box shape: the same bits
    for axis, side in (("X", 2), ("Y", 4), ("Z", 1)):
        monkeypatch.setenv("TETRA_BOX_" + axis, str(side))
    other = T.Plan(*n, nb, no, nw, mode=mode).dos(Et, Wt, omt)
    assert torch.equal(g, other)


@pytest.mark.parametrize("n,nb,no,dtype", [((1, 2, 1), 1, 1, "f32"), ((2, 3, 5), 3, 2, "f32"), ((31, 4, 4), 2, 4, "bf16"),
                                           ((32, 5, 3), 1, 8, "f16"), ((63, 2, 9), 2, 3, "f32"), ((6, 5, 7), 9, 1, "f32"),
                                           ((5, 4, 3), 40, 2, "f32")])
def test_fermi_level_shapes(T, n, nb, no, dtype):
    eps, w = bands(5, n, nb, no)
    eps *= 1.0 if n != (1, 2, 1) else 0.5
    plan = T.Plan(*n, nb, no, 16, weight_dtype=dtype)
    Et, Wt = tensors(plan, eps, w, n, plan.torch_weight_dtype)
    wr = from_layout(Et.cpu().numpy(), Wt.float().cpu().numpy(), *n, nb, no)[1]
    for filling in (0.13, 0.5, 0.77):
        target = filling * nb
        ef = plan.fermi_level(Et, Wt, target)
        below, above = (oracle.dos(eps, wr, *n, np.array([ef + d]), mode="integrated").sum() for d in (-1e-4, 1e-4))
        slack = 2.0 ** -7 * nb if dtype == "bf16" else 1e-5 * nb   # (rounded weights do not add up to one)
        assert below - slack <= target <= above + slack, (below, target, above)


@pytest.mark.parametrize("n,nb,no,nbins", [((4, 3, 5), 2, 1, 30), ((5, 4, 3), 3, 3, 7), ((3, 4, 6), 2, 5, 60),
                                           ((3, 3, 3), 2, 16, 50), ((4, 4, 4), 2, 16, 1200), ((6, 1, 2), 4, 4, 25)])
def test_dos_backward_shapes(T, n, nb, no, nbins):
    eps, w = bands(23, n, nb, no)
    edges = tbgen.bin_edges(float(eps.min()) + 0.5, float(eps.max()) - 0.5, nbins)   # some bands beyond both ends
    g = np.random.default_rng(2).normal(0, 1, (no, nbins)).astype(np.float32)
    plan = T.Plan(*n, nb, no, nbins, mode="bin")
    Et, Wt = tensors(plan, eps, w, n)
    ge = torch.empty_like(Et)
    gw = torch.empty(Wt.numel() + 1, device="cuda")[1:].view(Wt.shape)   # 4 bytes off a 16-byte boundary
    plan.dos_backward(Et, Wt, torch.from_numpy(edges).cuda(), torch.from_numpy(g).cuda(), ge, gw)
    a, b = from_layout(ge.cpu().numpy(), gw.cpu().numpy(), *n, nb, no)
    re, rw = oracle.dos_bin_grad(eps, w, *n, edges.astype(np.float64), g.astype(np.float64))
    close(b, rw, 1e-5)
    close(a, re, 1e-4)


@pytest.mark.parametrize("n,nb", [((2, 2, 2), 2), ((5, 3, 4), 3), ((6, 7, 5), 8)])
def test_susceptibility_shapes(T, n, nb):
    eps, w = bands(31, n, nb, 1)
    mu, q = float(np.median(eps)) + 0.05, (1, 2, 1)
    plan = T.Plan(*n, nb, 1, 16)
    Et, _ = tensors(plan, eps, w, n)
    e64 = eps.astype(np.float64)
    # a grid much wider than the tetrahedra (large contributions per energy) and a fine one
    for om in (tbgen.uniform_grid(-30.0, 30.0, 21), tbgen.uniform_grid(0.0, 9.0, 901)):
        for mode in ("point", "bin"):
            s = plan.spectral_t0(Et, q, mu, torch.from_numpy(om).cuda(), mode=mode)
            assert plan.spectral_status() == T.TETRA_OK
            close(s.cpu().numpy(), oracle.spectral_t0(e64, *n, q, mu, om.astype(np.float64), mode=mode), 2e-5)
    om = np.random.default_rng(1).permutation(tbgen.uniform_grid(-6.0, 12.0, 150))   # any order
    r = plan.chi0_real_t0(Et, q, mu, torch.from_numpy(om).cuda())
    close(r.cpu().numpy(), oracle.chi0_real_t0(e64, *n, q, mu, om.astype(np.float64)), 1e-4)
    # transition bands: rows of nb^2 values, whole vectors or not
    pair = T.Plan(*n, nb * nb, 1, 100)
    ep, wp = plan.pair_bands(Et, q, 0.05, mu, pair)
    re, rw = oracle.pair_bands(e64, *n, q, 0.05, mu)
    a, b = from_layout(ep.cpu().numpy(), wp.cpu().numpy(), *n, nb * nb, 1)
    close(a, re.reshape(a.shape), 1e-6)
    close(b, rw.reshape(b.shape), 1e-5)
