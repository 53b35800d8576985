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
