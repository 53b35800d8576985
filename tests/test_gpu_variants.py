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
