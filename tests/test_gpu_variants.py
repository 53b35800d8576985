"""The colour pass's compiled-in variants (whole groups of chains, one group only,
passes that record energies) and chain counts at their edges against the plain
path (needs a GPU): the states must be the same bits."""
import numpy as np
import pytest

import synthetic

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_1710_03038_gb300 as mpr  # noqa: E402


def images():
    """Odd sides, a tile that is all gap, a sparse and a one-tile image."""
    zs, gs = [], []
    for k, (h, w, f) in enumerate([(53, 37, 0.45), (33, 64, 0.1), (7, 9, 0.6)]):
        zs.append(synthetic.grf((h, w), nu=0.5, ell=6.0, mean=50, std=10, seed=40 + k).astype(np.float32))
        gs.append(synthetic.uniform_gaps((h, w), f, 50 + k).astype(np.uint8))
    gs[0][16:32, 16:32] = 1
    return zs, gs


def run(path, R, cg, model):
    zs, gs = images()
    ctx = mpr.Context(zs, gs, chains=R, params=mpr.Params(seed=77, path=path, chain_group=cg, model=model))
    ctx.set_T([0.2, 0.05, 0.4])
    ctx.sweep(3, "equil")
    ctx.sweep(1, "equil", record_energy=True)
    ctx.sweep(2, "measure")
    ctx.sweep(1, "measure", record_energy=True)
    info = ctx.chain_info()
    return ([s.cpu().numpy() for s in ctx.get_state()], info, [p.cpu().numpy() for p in ctx.predict()])


# (chains, group): one group only of 4, 8, 16 and 32 chains; several whole groups; one
# chain pair (slots 4 floats apart, 2 chains); a padded row; a group with missing pairs
@pytest.mark.parametrize("R,cg", [(4, 4), (8, 8), (16, 16), (32, 32), (8, 4), (64, 32), (2, 2), (1, 1),
                                  (31, 31), (20, 20), (36, 16)])
@pytest.mark.parametrize("model", ["mpr", "gmrf"])
def test_variants_equal_the_plain_path(R, cg, model):
    want, got = run("plain", R, cg, model), run("tiled", R, cg, model)
    for a, b in zip(got[0], want[0]):
        assert np.array_equal(a, b)
    for k in ("a", "accepted"):
        assert np.array_equal(got[1][k], want[1][k])
    # FP32 bond energies of up to 2e3 bonds, summed in other orders: 1e-6 of a bond
    assert np.allclose(got[1]["e_last"], want[1]["e_last"], rtol=0, atol=1e-6)
    # the mean of angles rounded to 2^-24 rad, mapped back and rounded to FP32
    for a, b in zip(got[2], want[2]):
        assert np.allclose(a, b, rtol=1e-6, atol=1e-5)


# ------------------------------------------------ launches per colour, resident runs
# Batches whose tiles and chain groups fit the GPU at once run their sweeps in one
# launch (the tests above); more than about a thousand blocks take a launch per colour.

def big_run(path, R, cg, model="mpr", n=2, hole=True):
    z = synthetic.grf((530, 545), nu=0.5, ell=9.0, mean=50, std=10, seed=61).astype(np.float32)
    g = synthetic.uniform_gaps((530, 545), 0.35, 62).astype(np.uint8)
    if hole:
        g[100:150, 200:260] = 1  # tiles that are all gap
    ctx = mpr.Context([z], [g], chains=R, params=mpr.Params(seed=78, path=path, chain_group=cg, model=model))
    ctx.set_T([0.1])
    ctx.sweep(n, "equil")
    ctx.sweep(1, "equil", record_energy=True)
    e = ctx.chain_info()["e_last"]
    ctx.sweep(n, "measure")
    info = ctx.chain_info()
    return ctx.get_state()[0], dict(info, e_last=e), ctx.predict()[0]


@pytest.mark.parametrize("R,cg,model", [(4, 4, "mpr"), (8, 8, "mpr"), (16, 16, "mpr"), (32, 32, "mpr"),
                                        (64, 32, "mpr"), (40, 32, "mpr"), (7, 7, "mpr"), (2, 2, "mpr"),
                                        (16, 16, "gmrf"), (24, 8, "gmrf")])
def test_launches_per_colour_equal_the_plain_path(R, cg, model):
    want, got = big_run("plain", R, cg, model), big_run("tiled", R, cg, model)
    assert torch.equal(got[0], want[0])
    for k in ("a", "accepted"):
        assert np.array_equal(got[1][k], want[1][k])
    assert np.allclose(got[1]["e_last"], want[1]["e_last"], rtol=0, atol=1e-6)
    assert torch.allclose(got[2], want[2], rtol=1e-6, atol=1e-5)


@pytest.mark.parametrize("R,model", [(4, "mpr"), (3, "mpr"), (8, "mpr"), (7, "gmrf"), (16, "mpr"), (13, "gmrf"),
                                     (32, "mpr"), (2, "mpr"), (20, "mpr"), (33, "gmrf")])
def test_small_groups_and_padded_rows_equal_the_plain_path(R, model):
    """Blocks of fewer warps (no tile is dense) and rows of 4, 8, 16 and 32 chains with up
    to half of them padding."""
    want, got = (big_run(p, R, 0, model, hole=False) for p in ("plain", "tiled"))
    assert torch.equal(got[0], want[0])
    for k in ("a", "accepted"):
        assert np.array_equal(got[1][k], want[1][k])
    assert torch.allclose(got[2], want[2], rtol=1e-6, atol=1e-5)


def small_ctx(path, R, seed=5, stream=None):
    zs, gs = images()
    ctx = mpr.Context(zs, gs, chains=R, params=mpr.Params(seed=seed, path=path), stream=stream)
    ctx.set_T([0.2, 0.05, 0.4], stream=stream)
    return ctx


@pytest.mark.parametrize("lengths", [(1, 1, 1, 1, 1, 1), (2, 4), (3, 3), (6,), (5, 1)])
@pytest.mark.parametrize("phase", ["equil", "measure"])
def test_resident_runs_join_without_a_seam(lengths, phase):
    """Six sweeps in runs of any length, states replaced in between by themselves: the
    plain path's states, acceptances and energies."""
    out = []
    for path, parts in (("plain", (6,)), ("tiled", lengths)):
        ctx = small_ctx(path, 10)
        ctx.sweep(2, "equil")
        for n in parts:
            ctx.set_state(ctx.get_state())
            ctx.sweep(n, phase, record_energy=True)
        out.append(([s.cpu().numpy() for s in ctx.get_state()], ctx.chain_info(), ctx.sweep_index()))
    for a, b in zip(out[0][0], out[1][0]):
        assert np.array_equal(a, b)
    assert np.array_equal(out[0][1]["accepted"], out[1][1]["accepted"])
    assert np.array_equal(out[0][1]["a"], out[1][1]["a"])
    assert np.allclose(out[0][1]["e_last"], out[1][1]["e_last"], rtol=0, atol=1e-6)
    assert out[0][2] == out[1][2]


@pytest.mark.parametrize("R,cg,model", [(8, 8, "mpr"), (7, 7, "gmrf"), (16, 16, "mpr"), (20, 16, "gmrf"), (32, 32, "mpr")])
def test_resident_and_launched_runs_alternate(R, cg, model):
    """A tile that is all gap: four warp steps and more, so that equilibration and recorded
    runs are launched per colour and sampling runs are resident (up to eight steps)."""
    out = []
    for path in ("plain", "tiled"):
        zs, gs = images()
        ctx = mpr.Context(zs, gs, chains=R, params=mpr.Params(seed=79, path=path, chain_group=cg, model=model))
        ctx.set_T([0.2, 0.05, 0.4])
        for n, phase, record in ((2, "equil", False), (3, "measure", False), (1, "measure", True),
                                 (2, "measure", False), (1, "equil", False), (2, "equil", True), (1, "measure", False)):
            ctx.sweep(n, phase, record_energy=record)
        out.append(([s.cpu().numpy() for s in ctx.get_state()], ctx.chain_info()))
    for a, b in zip(out[0][0], out[1][0]):
        assert np.array_equal(a, b)
    for k in ("a", "accepted"):
        assert np.array_equal(out[0][1][k], out[1][1][k])


def test_resident_runs_in_a_caller_capture_and_on_two_streams():
    """A captured run replays like a direct one, and contexts on two streams do not
    disturb each other."""
    want = []
    for seed in (5, 6):
        ctx = small_ctx("tiled", 10, seed)
        for _ in range(8):
            ctx.sweep(25, "measure")
        want.append([s.cpu().numpy() for s in ctx.get_state()])
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    ctxs = [small_ctx("tiled", 10, seed, stream=s) for seed, s in zip((5, 6), streams)]
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=streams[0]):
        ctxs[0].sweep(25, "measure", stream=streams[0])
    for _ in range(8):
        with torch.cuda.stream(streams[0]):
            graph.replay()
        ctxs[1].sweep(25, "measure", stream=streams[1])
    torch.cuda.synchronize()
    for ctx, w in zip(ctxs, want):
        for a, b in zip(ctx.get_state(), w):
            assert np.array_equal(a.cpu().numpy(), b)


# ------------------------------------------------------------------- dense views

@pytest.mark.parametrize("tile", [(16, 16), (32, 16), (32, 32)])
@pytest.mark.parametrize("R", [1, 33])
def test_dense_views_of_every_tile_shape(tile, R):
    """States, energies and predictions, one tile per block, against torch in FP64: ragged
    images, a tile that is all gap, one chain and a second group of chains."""
    zs, gs = images()
    ctx = mpr.Context(zs, gs, chains=R, params=mpr.Params(seed=9, tile=tile))
    ctx.set_T([0.2, 0.05, 0.4])
    start = ctx.get_state()
    gen = torch.Generator(device="cuda").manual_seed(4)
    new = [torch.rand(s.shape, device="cuda", generator=gen) * 6.28 for s in start]
    ctx.set_state(new)
    H = ctx.energy()
    for i, (s, n, g) in enumerate(zip(ctx.get_state(), new, gs)):
        gap = torch.from_numpy(g).cuda() != 0
        assert torch.equal(s[:, gap], n[:, gap])                   # gaps as set
        assert torch.equal(s[:, ~gap], start[i][:, ~gap])          # samples as mapped
        d = s.double()
        want = -(torch.cos(0.5 * (d[:, 1:] - d[:, :-1])).sum((1, 2)) +
                 torch.cos(0.5 * (d[:, :, 1:] - d[:, :, :-1])).sum((1, 2)))
        h, w = g.shape
        want /= h * (w - 1) + w * (h - 1)
        # FP32 differences and cosines of angles below 2 pi: 5e-7 a bond
        assert np.max(np.abs(H[i] - want.cpu().numpy())) < 5e-7
    ctx.sweep(5, "measure")
    s1, s2, n = ctx.accumulators()
    zh, sd = ctx.predict(std=True)
    info = ctx.image_info()
    for i, g in enumerate(gs):
        gap = torch.from_numpy(g).cuda() != 0
        scale = (float(info["zmax"][i]) - float(info["zmin"][i])) / (2 * np.pi)
        m = s1[i] / n
        want = torch.where(gap, float(info["zmin"][i]) + scale * m, torch.from_numpy(zs[i]).cuda().double())
        assert torch.equal(zh[i], want.float()) or (zh[i] - want.float()).abs().max() <= 4e-6 * want.abs().max()
        v = torch.sqrt((s2[i] / n - m * m).clamp(min=0)) * scale
        v = torch.where(gap, v, torch.zeros_like(v))
        # the variance is a difference of sums of up to 40 rad^2 in FP64 (1e-14): 1e-7 rad
        assert (sd[i].double() - v).abs().max() < 1e-6 * scale + 2e-7 * float(v.max())


@pytest.mark.parametrize("shape,R", [((128, 192), 32), ((131, 192), 33), ((100, 190), 32), ((97, 129), 40)])
def test_states_out_by_quads_and_by_pixels(shape, R):
    """States of more than 2^18 values: rows of whole quads (sides a multiple of four, whole
    and cut tiles) and of pixels; an output that starts off a 16-byte boundary."""
    h, w = shape
    z = synthetic.grf(shape, nu=0.5, ell=6.0, mean=50, std=10, seed=3).astype(np.float32)
    g = synthetic.uniform_gaps(shape, 0.4, 5).astype(np.uint8)
    g[16:32, 16:32] = 1
    out = []
    for path in ("plain", "tiled"):
        ctx = mpr.Context([z], [g], chains=R, params=mpr.Params(seed=5, path=path))
        out.append((ctx, ctx.get_state()[0]))
    assert torch.equal(out[0][1], out[1][1])
    from paper_1710_03038_gb300 import _lib
    flat = torch.full((R * h * w + 1,), -7.0, device="cuda")
    _lib.call("mpr_get_state", out[1][0]._ctx, mpr._ptr(flat[1:]), _lib.MPR_DEVICE, mpr._stream_ptr())
    torch.cuda.synchronize()
    assert float(flat[0]) == -7.0
    assert torch.equal(flat[1:].view(R, h, w), out[0][1])


# chains to a block 1, 2, 4, 8, 16 and 32, with and without lanes left over, and a last group
# of each width; fewer than 2^16 values by pixel, up to 151 tiles by strips, more by tiles
@pytest.mark.parametrize("R", [1, 2, 3, 4, 5, 8, 9, 16, 17, 31, 32, 33, 34, 36, 40, 48, 49])
@pytest.mark.parametrize("shape,tile,model", [((53, 37), (16, 16), "mpr"), ((150, 130), (16, 16), "mpr"),
                                              ((211, 203), (16, 16), "mpr"), ((211, 203), (16, 16), "gmrf"),
                                              ((520, 515), (32, 32), "mpr")])
def test_chain_energies_of_every_lane_split(R, shape, tile, model):
    """Energies of every chain against torch in FP64 on the states read back."""
    h, w = shape
    z = synthetic.grf(shape, nu=0.5, ell=6.0, mean=50, std=10, seed=7).astype(np.float32)
    g = synthetic.uniform_gaps(shape, 0.5, 8).astype(np.uint8)
    ctx = mpr.Context([z], [g], chains=R, params=mpr.Params(seed=9, tile=tile, model=model))
    d = ctx.get_state()[0].double()
    dx, dy = d[:, :, 1:] - d[:, :, :-1], d[:, 1:] - d[:, :-1]
    if model == "gmrf":
        want = sum((t * t / (2 * np.pi ** 2) - 1).sum((1, 2)) for t in (dx, dy))
    else:
        want = -sum(torch.cos(0.5 * t).sum((1, 2)) for t in (dx, dy))
    want /= h * (w - 1) + w * (h - 1)
    # FP32 differences and bonds of angles below 2 pi: 5e-7 a bond
    assert np.max(np.abs(ctx.energy()[0] - want.cpu().numpy())) < 5e-7


# either side of the line between the two ways (4.5 chains of a whole tile): few chains, a
# thin map with few pixels to a tile, more than one group of chains
@pytest.mark.parametrize("shape,R", [((256, 256), 4), ((256, 256), 5), ((512, 515), 1), ((20000, 3), 20),
                                     ((3, 20000), 40), ((20000, 3), 33)])
def test_states_in_and_out_by_tile_and_by_pixel(shape, R):
    z = synthetic.grf((64, 64), nu=0.5, ell=6.0, mean=50, std=10, seed=3).astype(np.float32)
    z = np.resize(z, shape)
    g = synthetic.uniform_gaps(shape, 0.4, 5).astype(np.uint8)
    gap = torch.from_numpy(g).cuda() != 0
    gen = torch.Generator(device="cuda").manual_seed(R)
    new = torch.rand(R, *shape, device="cuda", generator=gen) * 6.28
    out = []
    for path in ("plain", "tiled"):
        ctx = mpr.Context([z], [g], chains=R, params=mpr.Params(seed=5, path=path))
        start = ctx.get_state()[0]
        ctx.set_state([new])
        out.append((start, ctx.get_state()[0]))
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
    assert torch.equal(out[1][1][:, gap], new[:, gap])


@pytest.mark.parametrize("R,model", [(4, "mpr"), (3, "gmrf"), (8, "mpr"), (7, "mpr"), (16, "mpr"), (13, "gmrf")])
def test_blocks_of_fewer_warps_equal_the_plain_path(R, model):
    """1404 tiles: more than a wave of blocks, where small chain groups take fewer warps."""
    z = synthetic.grf((610, 575), nu=0.5, ell=9.0, mean=50, std=10, seed=63).astype(np.float32)
    g = synthetic.uniform_gaps((610, 575), 0.35, 64).astype(np.uint8)
    out = []
    for path in ("plain", "tiled"):
        ctx = mpr.Context([z], [g], chains=R, params=mpr.Params(seed=80, path=path, model=model))
        ctx.set_T([0.1])
        ctx.sweep(3, "equil")
        ctx.sweep(3, "measure")
        out.append((ctx.get_state()[0], ctx.chain_info(), ctx.predict()[0]))
    assert torch.equal(out[0][0], out[1][0])
    for k in ("a", "accepted"):
        assert np.array_equal(out[0][1][k], out[1][1][k])
    # the mean of angles rounded to 2^-24 rad, mapped back and rounded to FP32
    assert torch.allclose(out[0][2], out[1][2], rtol=1e-6, atol=1e-5)


@pytest.mark.parametrize("R", [4, 16])
def test_counting_passes_of_large_launches_equal_the_plain_path(R):
    """8281 tiles: the last sweep of a sampling run takes four warps, the others fewer."""
    z = np.resize(synthetic.grf((256, 256), nu=0.5, ell=9.0, mean=50, std=10, seed=65), (1450, 1449)).astype(np.float32)
    g = synthetic.uniform_gaps((1450, 1449), 0.3, 66).astype(np.uint8)
    out = []
    for path in ("plain", "tiled"):
        ctx = mpr.Context([z], [g], chains=R, params=mpr.Params(seed=81, path=path))
        ctx.set_T([0.1])
        ctx.sweep(1, "equil")
        ctx.sweep(1, "measure")
        ctx.sweep(2, "measure")
        out.append((ctx.get_state()[0], ctx.chain_info(), ctx.predict()[0]))
    assert torch.equal(out[0][0], out[1][0])
    assert np.array_equal(out[0][1]["accepted"], out[1][1]["accepted"])
    # the mean of angles rounded to 2^-24 rad, mapped back and rounded to FP32
    assert torch.allclose(out[0][2], out[1][2], rtol=1e-6, atol=1e-5)


def test_spread_of_the_smallest_and_largest_variances():
    """Restored sums far from any angle's: the spread is the square root of the variance, in
    FP64, for a map whose range makes it visible."""
    gen = torch.Generator(device="cuda").manual_seed(3)
    z = torch.rand(40, 48, device="cuda", generator=gen) * 1e28
    g = (torch.rand(40, 48, device="cuda", generator=gen) < 0.5).to(torch.uint8)
    ctx = mpr.Context([z], [g], chains=4, params=mpr.Params(seed=5))
    gap = g != 0
    var = 10.0 ** (80 * torch.rand(40, 48, dtype=torch.float64, device="cuda", generator=gen) - 48)
    var[0] = 0.0
    ctx.set_accumulators([torch.zeros_like(var)], [var * 8], 8)
    sd = ctx.predict(std=True)[1][0]
    info = ctx.image_info()
    want = (torch.sqrt(var) * (float(info["zmax"][0]) - float(info["zmin"][0])) / (2 * np.pi))[gap]
    # FP64 throughout and one rounding to FP32 (infinite beyond its range)
    over = torch.isinf(want.float())
    assert torch.isinf(sd[gap][over]).all()
    assert ((sd[gap].double() - want)[~over].abs() <= 1.2e-7 * want[~over]).all()
