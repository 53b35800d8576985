"""Resident runs of sweeps (one launch per run) against launches per colour, bit for bit
(needs a GPU).  An image of a batch too large for the GPU at once is launched per colour;
alone it is resident.  Its random stream and its arithmetic are the same in both."""
import numpy as np
import pytest

import synthetic

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_1710_03038_gb300 as mpr  # noqa: E402


def image(shape, frac, seed):
    z = synthetic.grf(shape, nu=0.5, ell=6.0, mean=50, std=10, seed=seed).astype(np.float32)
    return z, synthetic.uniform_gaps(shape, frac, seed + 1).astype(np.uint8)


def context(images, R, cg, T=0.1, **kw):
    ctx = mpr.Context([z for z, _ in images], [g for _, g in images], chains=R,
                      params=mpr.Params(seed=91, chain_group=cg, **kw))
    ctx.set_T(T)
    return ctx


FILLER = ((530, 545), 0.3, 201)  # 1190 tiles: more than one wave of blocks


# red and black counts of the tiles between 10 and 90: the flush of a tile's sums crosses
# every boundary of its 128 threads
@pytest.mark.parametrize("R,cg,frac", [(8, 8, 0.4), (16, 16, 0.4), (6, 6, 0.45), (24, 8, 0.4), (32, 32, 0.3)])
@pytest.mark.parametrize("model", ["mpr", "gmrf"])
def test_sums_of_sampling_runs(R, cg, frac, model):
    """The realisation sums of runs of every length, many times over, to the last bit."""
    img = image((130, 147), frac, 11)
    alone = context([img], R, cg, model=model)
    launched = context([img, image(*FILLER)], R, cg, model=model)
    for n in (1, 2, 3, 1, 7, 1, 2, 5, 1, 4) * 3:
        alone.sweep(n, "measure")
        launched.sweep(n, "measure")
        got, want = alone.accumulators(), launched.accumulators()
        assert torch.equal(got[0][0], want[0][0])
        assert torch.equal(got[1][0], want[1][0])
    assert torch.equal(alone.get_state()[0], launched.get_state()[0])


# ------------------------------------------------------------------ a wait that gives up

def device_error(call):
    with pytest.raises(mpr._lib.MprError) as e:
        call()
    assert e.value.status == 8


# (states of 1.5e5 values go out by pixel, of 3e5 by tile)
@pytest.mark.parametrize("R,phase", [(8, "equil"), (8, "measure"), (16, "measure")])
def test_a_run_that_gives_up_is_reported(R, phase):
    """A wait limit of 0: every wait gives up.  Calls that return host values fail; what goes
    to device memory is NaN at the gaps; the context stays unusable, others are not touched."""
    z, g = image((130, 147), 0.3, 31)
    gap, smp = torch.from_numpy(g).cuda() != 0, torch.from_numpy(z).cuda()
    ctx = context([(z, g)], R, 8)
    ctx.sweep(2, "measure")
    ctx.check()
    ctx.set_wait_limit(0)
    ctx.sweep(3, phase)
    zh, sd = ctx.predict(std=True)
    s1, s2, _ = ctx.accumulators()
    for t in (zh[0], sd[0], s1[0], s2[0], *ctx.get_state()[0]):
        assert bool(torch.isnan(t[gap]).all()) and not bool(torch.isnan(t[~gap]).any())
    assert torch.equal(zh[0][~gap], smp[~gap])
    device_error(ctx.check)
    device_error(ctx.energy)
    device_error(ctx.chain_info)
    device_error(ctx.get_T)
    device_error(ctx.energy_history)
    device_error(lambda: ctx.predict_host(torch.empty(z.size)))
    ctx.set_wait_limit(1 << 21)
    ctx.set_sweep_index(0, 0)  # (does not hide it)
    device_error(ctx.check)
    again = context([(z, g)], R, 8)
    again.sweep(3, phase)
    again.check()


def test_a_temperature_that_gives_up_is_reported():
    z, g = image((130, 147), 0.3, 31)
    ctx = mpr.Context([z], [g], chains=4)
    ctx.set_wait_limit(0)
    device_error(ctx.estimate_T)
    ctx = mpr.Context([z], [g], chains=4)
    ctx.set_wait_limit(0)
    ctx.estimate_T_async()
    ctx.set_wait_limit(1 << 21)
    ctx.sweep(2, "measure")
    assert bool(torch.isnan(ctx.predict()[0][torch.from_numpy(g).cuda() != 0]).all())
    device_error(ctx.check)


# ------------------------------------------------------------------ what was launched

def kernels(call):
    before = mpr.launch_count()
    call()
    return mpr.launch_count() - before


@pytest.mark.parametrize("use_graphs", [True, False])
def test_launch_count(use_graphs):
    """One kernel for a resident run; two passes and the bookkeeping for a launched sweep, the
    bookkeeping once for sampling sweeps without energies; replays like the launches."""
    img, side = image((130, 147), 0.3, 41), torch.cuda.Stream()
    with torch.cuda.stream(side):
        alone = context([img], 8, 8, use_graphs=use_graphs)
        big = context([img, image(*FILLER)], 8, 8, use_graphs=use_graphs)
        plain = context([img], 8, 0, path="plain")
        assert big.sweep_launches()[0] == 3
        for n in (1, 5, 5):
            assert kernels(lambda: alone.sweep(n, "measure")) == 1
            assert kernels(lambda: alone.sweep(n, "equil")) == 1
            assert kernels(lambda: big.sweep(n, "measure")) == 2 * n + 1
            assert kernels(lambda: big.sweep(n, "equil")) == 3 * n
            assert kernels(lambda: big.sweep(n, "measure", record_energy=True)) == 3 * n
            assert kernels(lambda: plain.sweep(n, "measure")) == 3 * n
        # (per sweep the stop rule's kernel too)
        done = []
        got = kernels(lambda: done.append(big.equilibrate(i_max=30)))
        assert got == 4 * done[0]
        assert kernels(lambda: big.predict()) == 1
        assert kernels(lambda: big.image_info()) == 0
    assert kernels(lambda: context([img], 8, 8)) > 20


# tiles per image: 484 (two runs fit the GPU at once), 361 and 625 (one does), 90
@pytest.mark.parametrize("shape,R,frac,want", [
    ((130, 147), 8, 0.3, dict(equil=1, measure=1, equil_rec=1, measure_rec=1, single_rec=1)),
    ((350, 350), 4, 0.4, dict(equil=1, measure=1, equil_rec=1, measure_rec=1, single_rec=0)),
    ((300, 300), 16, 0.2, dict(equil=0, measure=1, equil_rec=0, measure_rec=1, single_rec=0)),
    ((400, 400), 8, 0.2, dict(equil=0, measure=1, equil_rec=0, measure_rec=1, single_rec=0)),
])
def test_which_runs_are_resident(shape, R, frac, want):
    ctx = context([image(shape, frac, 51)], R, 0)
    got = {}
    for name, n, phase, record in (("equil", 3, "equil", False), ("measure", 3, "measure", False),
                                   ("equil_rec", 3, "equil", True), ("measure_rec", 3, "measure", True),
                                   ("single_rec", 1, "equil", True)):
        got[name] = int(kernels(lambda: ctx.sweep(n, phase, record_energy=record)) == 1)
    assert got == want


# more than 64 tiles to an image: several words to a chain, recorders of many packets;
# chain groups of 4 with and without a rest, one group of all chains
@pytest.mark.parametrize("shape,R,model", [((350, 350), 4, "mpr"), ((256, 256), 16, "mpr"), ((250, 250), 10, "mpr"),
                                           ((251, 173), 16, "gmrf"), ((300, 300), 6, "gmrf")])
def test_images_of_many_tiles(shape, R, model):
    img, other = image(shape, 0.4, 61), image(FILLER[0], 0.3, 71)
    out = []
    for images, cg in (([img], 0), ([img, other], 4)):
        ctx = context(images, R, cg, model=model)
        if len(images) == 1:
            assert kernels(lambda: ctx.sweep(2, "measure")) == 1
        else:
            ctx.sweep(2, "measure")
        records = []
        for n, phase, record in ((3, "equil", False), (4, "equil", True), (3, "measure", True), (5, "measure", False),
                                 (1, "equil", True)):
            ctx.sweep(n, phase, record_energy=record)
            info = ctx.chain_info()
            records.append({k: v[0] for k, v in info.items()})
        out.append((ctx.get_state()[0], ctx.accumulators(), records))
    assert torch.equal(out[0][0], out[1][0])
    assert torch.equal(out[0][1][0][0], out[1][1][0][0]) and torch.equal(out[0][1][1][0], out[1][1][1][0])
    for a, b in zip(out[0][2], out[1][2]):
        assert np.array_equal(a["a"], b["a"]) and np.array_equal(a["accepted"], b["accepted"])
        # the tiles' sums are the same bits; their FP64 total in another order
        assert np.allclose(a["e_last"], b["e_last"], rtol=0, atol=1e-10, equal_nan=True)


# ------------------------------------------------------------------ graphs of launches

@pytest.mark.parametrize("R,hole", [(6, False), (36, False), (8, True)])
def test_replayed_graphs_of_a_launched_batch(R, hole):
    """A batch that is launched per colour: runs captured once and replayed (also sampling runs,
    whose launches carry their place in the run and share one bookkeeping launch) give the
    bits of direct launches.  36 chains leave a group of 4 to a launch of its own, a hole
    makes heavy tiles."""
    z, g = image((530, 545), 0.35, 81)
    if hole:
        g[100:160, 200:270] = 1
    side, out = torch.cuda.Stream(), []
    for use_graphs in (True, False):
        with torch.cuda.stream(side):
            ctx = context([(z, g)], R, 32 if R > 32 else 0, use_graphs=use_graphs)
            assert kernels(lambda: ctx.sweep(6, "equil")) >= 18
            for n, phase, record in ((5, "measure", False), (5, "measure", False), (6, "equil", True),
                                     (5, "measure", False), (7, "measure", True), (6, "equil", True),
                                     (7, "measure", True), (5, "measure", False)):
                ctx.sweep(n, phase, record_energy=record)
            ctx.sweep(7, "measure", record_energy=True)
            out.append((ctx.get_state()[0], ctx.accumulators(), ctx.chain_info(), ctx.sweep_index()))
        side.synchronize()
    assert torch.equal(out[0][0], out[1][0])
    assert torch.equal(out[0][1][0][0], out[1][1][0][0]) and torch.equal(out[0][1][1][0], out[1][1][1][0])
    assert np.array_equal(out[0][2]["a"], out[1][2]["a"]) and np.array_equal(out[0][2]["accepted"], out[1][2]["accepted"])
    # FP64 totals of the tiles' sums, added in any order
    assert np.allclose(out[0][2]["e_last"], out[1][2]["e_last"], rtol=0, atol=1e-10)
    assert out[0][3] == out[1][3]
