"""The double step of thin columns and the float step at the edges of their
tiles, and captured steps across a change of geometry."""
import numpy as np
import pytest

from paper_2510_18688_gb300 import workloads as W

FIELDS = ("phi", "fs", "fl", "T", "rhoH", "p", "ux", "uy", "rho", "mu", "w", "mdot")


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from oracle import oracle as O
    from paper_2510_18688_gb300 import build, lbm
    build.build()
    lbm.load()
    return O, lbm


def _close64(got, ref):  # the parity bar of the FP64 step
    for k in FIELDS:
        scale = max(np.abs(ref[k]).max(), 1e-300)
        assert np.abs(got[k] - ref[k]).max() <= 1e-10 * scale + 1e-18, k


# columns: rows below, at and above a warp's 32 nodes, with and without rows
# whose 32 x 8 tile lies inside the grid
@pytest.mark.gpu
@pytest.mark.parametrize("nx,ny", [(31, 2), (32, 8), (33, 5), (64, 16), (97, 24), (129, 31)])
@pytest.mark.parametrize("seed", [0, 1, 2, 3])
@pytest.mark.parametrize("diag_every", [0, 4])
def test_columns_match_the_oracle(env, nx, ny, seed, diag_every):
    O, lbm = env
    cfg, arr = W.random_state(nx, ny, seed=seed)
    ref = O.from_workload((cfg, arr)).step(21).fields()
    s = lbm.Solver(cfg, precision="fp64", diag_every=diag_every).set_geometry(arr).step(21)
    _close64(s.fields(), ref)
    s.close()


# the one-dimensional columns, whose velocity across is rounding alone: the four
# warps a tile give every bit of step_tile, which forms 4 and 5 are
@pytest.mark.gpu
@pytest.mark.parametrize("wl", [W.neumann(400, 4), W.stefan(512, 8), W.stefan(300, 5)],
                         ids=["neumann400x4", "stefan512x8", "stefan300x5"])
def test_columns_keep_the_bits_of_the_fused_tile(env, wl, monkeypatch):
    _, lbm = env
    got = {}
    for form in ("0", "4", "5"):
        monkeypatch.setenv("LBM_KERNEL_FORM", form)
        s = lbm.Solver(wl[0], precision="fp64").set_geometry(wl[1])
        got[form] = [s.step(n).fields() for n in (1, 15, 184)]
        s.close()
    for form in ("4", "5"):
        for x, y in zip(got["0"], got[form]):
            for k in FIELDS:
                assert np.array_equal(x[k], y[k]), (form, k)


@pytest.mark.gpu
@pytest.mark.parametrize("lattices", [1, 2, 4, 3, 5, 6, 7])
def test_columns_lattice_sets_and_the_readings_variant(env, lattices):
    O, lbm = env
    cfg, arr = W.random_state(75, 11, seed=3, lattices=lattices)
    cfg = dict(cfg, readings=1, gx=3e-6, gy=-2e-6)
    ref = O.from_workload((cfg, arr)).step(25).fields()
    s = lbm.Solver(cfg, precision="fp64").set_geometry(arr).step(25)
    _close64(s.fields(), ref)
    s.close()


# the float step's 32 x 8 tiles: one short, whole and one node over, in every
# kernel form, with every kind of wall
@pytest.mark.gpu
@pytest.mark.parametrize("nx,ny", [(31, 31), (32, 32), (33, 33), (63, 41), (65, 40)])
@pytest.mark.parametrize("seed", [0, 1, 2, 3])
@pytest.mark.parametrize("form", [0, 2, 3, 4, 5])
def test_float_forms_match_the_oracle(env, nx, ny, seed, form, monkeypatch):
    O, lbm = env
    monkeypatch.setenv("LBM_KERNEL_FORM", str(form))
    cfg, arr = W.random_state(nx, ny, seed=seed)
    ref = O.from_workload((cfg, arr)).step(21).fields()
    s = lbm.Solver(cfg, precision="fp32", diag_every=4).set_geometry(arr).step(21)
    got = s.fields()
    for k in FIELDS:
        a, b = ref[k], got[k]
        den = max(np.linalg.norm(a), 1e-30 * np.sqrt(a.size))
        assert np.linalg.norm(a - b) <= 1e-4 * den or \
            np.abs(a - b).max() <= 1e-6 * max(np.abs(a).max(), 1e-3), k
    s.close()


@pytest.mark.gpu
@pytest.mark.parametrize("prec", ["fp32", "fp16s", "fp64"])
def test_captured_steps_across_geometries_with_and_without_a_mask(env, prec):
    """Periods captured for one geometry serve the next; a mask that comes or
    goes is seen: bit for bit a fresh context."""
    _, lbm = env
    cfg, arr = W.random_state(70, 40, seed=1)
    other = W.random_state(70, 40, seed=5)[1]
    bare = {k: v for k, v in other.items() if k != "mask"}
    assert arr["mask"].any()
    s = lbm.Solver(cfg, precision=prec, diag_every=4)
    for a in (arr, other, bare, arr, bare):
        got = s.set_geometry(a).step(100).fields()
        f = lbm.Solver(cfg, precision=prec, diag_every=4).set_geometry(a).step(100)
        want = f.fields()
        for k in FIELDS:
            assert np.array_equal(got[k], want[k], equal_nan=True), k
        f.close()
    s.close()
