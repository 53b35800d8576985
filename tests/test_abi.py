"""The C ABI: the library builds for sm_103a, loads, and exports every declared symbol.

No compute call is made here: these run without a GPU.
"""
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _declared_functions():
    with open(os.path.join(ROOT, "include", "mpr.h")) as f:
        src = f.read()
    src = re.sub(r"/\*.*?\*/", "", src, flags=re.S)
    names = set(re.findall(r"\b(mpr_[A-Za-z0-9_]+)\s*\(", src))
    return sorted(names)


@pytest.fixture(scope="module")
def lib():
    from paper_1710_03038_gb300 import build
    build.build()
    from paper_1710_03038_gb300 import _lib
    return _lib.load()


def test_header_declares_the_five_method_entry_points():
    names = _declared_functions()
    for n in ("mpr_init_grid", "mpr_estimate_T", "mpr_sweep", "mpr_energy", "mpr_predict"):
        assert n in names


def test_library_exports_every_declared_symbol(lib):
    missing = [n for n in _declared_functions() if not hasattr(lib, n)]
    assert not missing, missing


def test_binding_covers_every_declared_symbol():
    from paper_1710_03038_gb300 import _lib
    assert set(_declared_functions()) <= set(_lib.EXPORTS)


def test_host_only_calls(lib):
    """Calls that touch no device: defaults, status strings, workspace sizing, argument errors."""
    import ctypes as C
    from paper_1710_03038_gb300 import _lib
    p = _lib.MprParams()
    assert lib.mpr_default_params(C.byref(p)) == 0
    assert (p.q, p.J, p.A_targ, p.k_a) == (0.5, 1.0, 0.3, 3.0)
    o = _lib.MprTOpts()
    assert lib.mpr_default_T_opts(C.byref(o)) == 0
    assert lib.mpr_status_string(0) == b"ok"
    Lx = _lib.int_array([64, 37])
    Ly = _lib.int_array([64, 53])
    nbytes = C.c_size_t()
    assert lib.mpr_workspace_size(2, Lx, Ly, None, 4, C.byref(p), None, C.byref(nbytes)) == 0
    worst = nbytes.value
    ng = _lib.i64_array([1000, 500])
    assert lib.mpr_workspace_size(2, Lx, Ly, ng, 4, C.byref(p), None, C.byref(nbytes)) == 0
    assert 0 < nbytes.value < worst
    # invalid arguments are rejected on the host
    bad = _lib.int_array([1, 37])
    assert lib.mpr_workspace_size(2, bad, Ly, None, 4, C.byref(p), None, C.byref(nbytes)) == 1
    assert lib.mpr_workspace_size(2, Lx, Ly, None, 0, C.byref(p), None, C.byref(nbytes)) == 1
    p.q = 0.7
    assert lib.mpr_workspace_size(2, Lx, Ly, None, 4, C.byref(p), None, C.byref(nbytes)) == 1
    assert b"q" in lib.mpr_last_error()
    out = C.c_void_p()
    p.q = 0.5
    # NULL inputs are rejected before any device work
    assert lib.mpr_init_grid(C.byref(out), 2, Lx, Ly, 4, C.byref(p), None, None, None, 0, None, 0,
                             None) == 1
    # cross-validated q: workspace sizing and argument checks, all before any device work
    qb = C.c_size_t()
    assert lib.mpr_select_q_workspace_size(64, 64, 8, C.byref(p), None, C.byref(qb)) == 0
    assert lib.mpr_workspace_size(1, _lib.int_array([64]), _lib.int_array([64]), None, 8,
                                  C.byref(p), None, C.byref(nbytes)) == 0
    assert qb.value > nbytes.value  # one context plus the staged inputs
    dummy = C.c_void_p(256)          # never dereferenced: the checks below fail first
    qs = (C.c_double * 2)(0.25, 0.6)
    sc = (C.c_double * 2)()
    assert lib.mpr_select_q(64, 64, dummy, dummy, dummy, 0, 2, qs, 8, 10, 10, C.byref(p), None,
                            dummy, qb, sc, None, None, None) == 1
    assert b"(0, 1/2]" in lib.mpr_last_error()
    qs[1] = 0.5
    assert lib.mpr_select_q(64, 64, dummy, dummy, dummy, 0, 2, qs, 8, 10, 0, C.byref(p), None,
                            dummy, qb, sc, None, None, None) == 1
    p.model = 1
    assert lib.mpr_select_q(64, 64, dummy, dummy, dummy, 0, 2, qs, 8, 10, 10, C.byref(p), None,
                            dummy, qb, sc, None, None, None) == 1
    assert b"MPR bond" in lib.mpr_last_error()
    p.model = 0


def test_no_cpu_fallback_in_product_package():
    """The package never imports the oracle (the CPU reference is test infrastructure)."""
    pkg = os.path.join(ROOT, "paper_1710_03038_gb300")
    for dirpath, _, files in os.walk(pkg):
        for fn in files:
            if fn.endswith((".py", ".cu", ".cuh", ".h", ".cpp")):
                with open(os.path.join(dirpath, fn)) as f:
                    text = f.read()
                assert "import oracle" not in text and "from oracle" not in text, fn
                assert "mpr_oracle" not in text, fn


def _workspace(lib, side, chains, images=1, **fields):
    import ctypes as C
    from paper_1710_03038_gb300 import _lib
    p = _lib.MprParams()
    lib.mpr_default_params(C.byref(p))
    for k, v in fields.items():
        setattr(p, k, v)
    L, n = _lib.int_array([side] * images), C.c_size_t()
    assert lib.mpr_workspace_size(images, L, L, None, chains, C.byref(p), None, C.byref(n)) == 0
    return n.value


@pytest.mark.parametrize("chains", [1, 4, 10, 32, 100])
@pytest.mark.parametrize("side", [64, 200, 333, 512, 700, 1024, 1400])
def test_the_smallest_tiles_need_the_largest_workspace(lib, side, chains):
    """What mpr_autotune asks its callers to rely on: a workspace for 16 x 16 tiles holds
    every candidate."""
    for images in (1, 3):
        want = _workspace(lib, side, chains, images, tile_x=16, tile_y=16)
        assert _workspace(lib, side, chains, images, tile_x=32, tile_y=16) <= want
        assert _workspace(lib, side, chains, images, tile_x=32, tile_y=32) <= want


@pytest.mark.parametrize("side,chains", [(700, 32), (520, 64), (530, 4)])
def test_batches_that_cannot_be_resident_reserve_no_packets(lib, side, chains):
    """More than 1064 blocks (152 SMs of seven), or the printed over-relaxation: 16 x 16 tiles
    need what their slots and lists add to those of 32 x 32 tiles, and no packets."""
    tiles = (-(-side // 16)) ** 2
    for fields in (dict(), dict(literal_or=1)):
        extra = (_workspace(lib, side, chains, tile_x=16, tile_y=16, **fields)
                 - _workspace(lib, side, chains, tile_x=32, tile_y=32))
        # 8 slots of padding, their records, the ring lists and the tile's own records
        assert extra < tiles * (8 * (4 * ((chains + 31) // 32 * 32) + 64) + 1024)
    assert (_workspace(lib, 128, 32, tile_x=16, tile_y=16, literal_or=1)
            < _workspace(lib, 128, 32, tile_x=16, tile_y=16))


@pytest.mark.parametrize("chains", [5, 9, 17, 21, 33, 36, 40, 65, 100])
def test_states_are_rounded_by_less_than_a_third(lib, chains):
    """A workspace's states: within 30 % of 4 bytes per chain and pixel (and 4 chains)."""
    side = 1024
    states = _workspace(lib, side, chains) - _workspace(lib, side, 1)
    assert states <= 4.0 * side * side * (1.3 * chains + 4) + 2 ** 24
