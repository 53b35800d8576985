"""Lattice energies and gradients against torch in FP64, on either side of the line between
a thread per pixel and a thread per column (needs a GPU): single pixels, thin grids, whole
and cut blocks of columns and rows, more than one launch of grids, ragged batches."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_1710_03038_gb300 as mpr  # noqa: E402
from paper_1710_03038_gb300 import _lib  # noqa: E402

J, Q = 1.25, 0.35


def exact(phi, w):
    """H, dL/dphi and dL/dJ of one grid, L = w H."""
    d = phi.double()
    dx, dy = Q * (d[:, 1:] - d[:, :-1]), Q * (d[1:] - d[:-1])
    B = float(torch.cos(dx).sum() + torch.cos(dy).sum())
    g = torch.zeros_like(d)
    g[:, 1:] += torch.sin(dx)
    g[:, :-1] -= torch.sin(dx)
    g[1:] += torch.sin(dy)
    g[:-1] -= torch.sin(dy)
    return -J * B, w * J * Q * g, -w * B


@pytest.mark.parametrize("shapes", [
    [(1, 1)], [(2, 3)], [(64, 64)], [(1, 700)], [(700, 1)], [(200000, 2)], [(2, 200000)], [(5000, 33)],
    [(512, 400)], [(449, 511)], [(17, 129)] * 100, [(33, 31)] * 300, [(130, 129)] * 12,
    [(40, 40), (700, 300), (1, 5), (300, 700)], [(1500, 1450)], [(16, 128)] * 1000,
])
def test_energies_and_gradients(shapes):
    n = len(shapes)
    gen = torch.Generator(device="cuda").manual_seed(n)
    sizes = [h * w for h, w in shapes]
    phi = 6.28 * torch.rand(sum(sizes), device="cuda", generator=gen)
    w = torch.randn(n, dtype=torch.float64, device="cuda", generator=gen)
    lx, ly = _lib.int_array([s[1] for s in shapes]), _lib.int_array([s[0] for s in shapes])
    H = torch.full((n,), 7.0, dtype=torch.float64, device="cuda")
    torque, grad = torch.full_like(phi, 7.0), torch.full_like(phi, 7.0)
    gJ, gJ2 = torch.full((1,), 7.0, dtype=torch.float64, device="cuda"), torch.full((1,), 7.0, dtype=torch.float64, device="cuda")
    p, s = mpr._ptr, mpr._stream_ptr()
    _lib.call("mpr_lattice_energy", n, lx, ly, p(phi), Q, J, p(H), s)
    _lib.call("mpr_lattice_torque", n, lx, ly, p(phi), Q, J, p(w), p(torque), s)
    _lib.call("mpr_lattice_grad", n, lx, ly, p(phi), Q, J, p(w), p(grad), p(gJ), s)
    _lib.call("mpr_lattice_grad", n, lx, ly, p(phi), Q, J, p(w), None, p(gJ2), s)
    off, want_J, tol_J = 0, 0.0, 1e-12
    for k, (shape, m) in enumerate(zip(shapes, sizes)):
        h, g, j = exact(phi[off:off + m].view(shape), float(w[k]))
        bonds = shape[0] * (shape[1] - 1) + shape[1] * (shape[0] - 1)
        # a bond's FP32 term: the difference, its product with q and the function, 5e-7 at most
        assert abs(float(H[k]) - h) <= 5e-7 * J * bonds + 1e-12
        for t in (torque, grad):
            assert float((t[off:off + m].view(shape).double() - g).abs().max()) <= 4 * 5e-7 * J * Q * abs(float(w[k])) + 1e-30
        want_J += j
        tol_J += 5e-7 * abs(float(w[k])) * bonds
        off += m
    assert abs(float(gJ) - want_J) <= tol_J and abs(float(gJ2) - want_J) <= tol_J


@pytest.mark.parametrize("lx,ly", [(2 ** 31 - 1, 1), (1, 2 ** 31 - 1)])
def test_the_longest_lines(lx, ly):
    """A constant line of 2^31 - 1 pixels: every bond is 1."""
    phi = torch.full((2 ** 31 - 1,), 3.0, device="cuda")
    H = torch.empty(1, dtype=torch.float64, device="cuda")
    _lib.call("mpr_lattice_energy", 1, _lib.int_array([lx]), _lib.int_array([ly]), mpr._ptr(phi), Q, 1.0,
              mpr._ptr(H), mpr._stream_ptr())
    assert float(H) == -(2.0 ** 31 - 2)


@pytest.mark.parametrize("big", [1e37, 1e-33])
def test_energies_of_extreme_exchange(big):
    """J near the ends of FP32: the sums of energies scale with J (FP32 terms, wider sums).
    Every sum that is kept in two FP32 words: grids by column, the sample energy of a
    context and of the allocation-free entry point, the chains' energies by tile."""
    gen = torch.Generator(device="cuda").manual_seed(5)
    phi = 6.28 * torch.rand(1, 600, 513, device="cuda", generator=gen)
    z = 50 + 10 * torch.randn(211, 203, device="cuda", generator=gen)
    g = (torch.rand(211, 203, device="cuda", generator=gen) < 0.4).to(torch.uint8)
    got = []
    for j in (1.0, big):
        H = mpr.lattice_energy(phi, q=Q, J=j)
        ns = mpr.sample_energy_noalloc([z], [g], J=j)["e_s"]
        out = [H.cpu().numpy(), ns.cpu().numpy()]
        for model in ("mpr", "gmrf"):
            ctx = mpr.Context([z], [g], chains=10, params=mpr.Params(J=j, model=model, seed=4))
            out += [ctx.image_info()["e_s"], ctx.energy().reshape(-1)]
        got.append(out)
    for k, (a, b) in enumerate(zip(*got)):
        # J and every bond's product with it are rounded to FP32 once each, 6e-8 of a bond; the
        # first is a sum over bonds, the others are means
        assert abs(b / big - a).max() <= 1.2e-7 * (2 * phi.numel() if k == 0 else 1)
