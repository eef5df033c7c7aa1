"""The double-precision node step: grids at the edges of its warps, blocks and
of the rule that leaves one-dimensional columns to the fused tile; batches that mix
the two; the reciprocal its kernels take."""
from fractions import Fraction

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


def _close(got, ref, tol=1e-10):  # the parity bar of the FP64 step
    for k in FIELDS:
        scale = max(np.abs(ref[k]).max(), 1e-300)
        assert np.abs(got[k] - ref[k]).max() <= tol * scale + 1e-18, k


# columns of one warp and less, rows that end inside a warp and a block, and
# both sides of the rule for one-dimensional columns
SIZES = [(2, 32), (3, 33), (31, 32), (32, 32), (33, 32), (33, 31), (64, 64), (129, 33), (40, 200),
         (1057, 31), (1060, 31), (701, 39)]


@pytest.mark.gpu
@pytest.mark.parametrize("nx,ny", SIZES)
@pytest.mark.parametrize("seed", [0, 3])
def test_sizes_match_the_oracle(env, nx, ny, seed):
    O, lbm = env
    cfg, arr = W.random_state(nx, ny, seed=seed)
    steps = 21
    o = O.from_workload((cfg, arr)).step(steps - 1)
    rd = o.diagnostics()
    s = lbm.Solver(cfg, precision="fp64", diag_every=1).set_geometry(arr).step(steps)
    d = s.diagnostics(compute=False)
    _close(s.fields(), o.step(1).fields())
    for k, v in rd.items():
        if k != "step":
            assert abs(d[k] - v) <= 1e-12 * (abs(v) + nx * ny), k
    s.close()


# (columns take the fused tile, whose copies with and without sums
# round some nodes differently)
@pytest.mark.gpu
@pytest.mark.parametrize("nx,ny", [z for z in SIZES if z[1] >= 32])
@pytest.mark.parametrize("seed", [0, 3])
def test_fused_sums_equal_the_read_out(env, nx, ny, seed):
    """The read-out's sums of a state are those fused into the step that read
    it, and steps with and without sums give the same state, bit for bit."""
    _, lbm = env
    cfg, arr = W.random_state(nx, ny, seed=seed)
    s = lbm.Solver(cfg, precision="fp64", diag_every=1).set_geometry(arr).step(21)
    t = lbm.Solver(cfg, precision="fp64").set_geometry(arr).step(20)
    assert t.diagnostics() == s.diagnostics(compute=False)
    s.close()
    t.close()


@pytest.mark.gpu
@pytest.mark.parametrize("lattices", [1, 2, 4, 3, 5, 6, 7])
def test_lattice_sets_and_the_readings_variant(env, lattices):
    O, lbm = env
    cfg, arr = W.random_state(45, 37, seed=3, lattices=lattices)
    cfg = dict(cfg, readings=1, gx=3e-6, gy=-2e-6)
    ref = O.from_workload((cfg, arr)).step(25).fields()
    s = lbm.Solver(cfg, precision="fp64").set_geometry(arr).step(25)
    _close(s.fields(), ref)
    s.close()


@pytest.mark.gpu
def test_batch_of_columns_and_wide_grids_equals_single_grids(env):
    """Each grid of a batch takes the kernel lbm_step takes: bit for bit."""
    _, lbm = env
    wls = [W.stefan(130, 5), W.random_state(40, 33, seed=1), W.random_state(50, 31, seed=2),
           W.random_state(33, 64, seed=3)]
    ss = [lbm.Solver(c, precision="fp64", diag_every=3).set_geometry(a) for c, a in wls]
    b = lbm.Batch(ss).step(7).step(33)
    for (cfg, arr), s in zip(wls, ss):
        alone = lbm.Solver(cfg, precision="fp64", diag_every=3).set_geometry(arr).step(40)
        fa, fb = alone.fields(), s.fields()
        for k in FIELDS:
            assert np.array_equal(fa[k], fb[k]), k
        assert alone.diagnostics(compute=False) == s.diagnostics(compute=False)
        alone.close()
    b.close()


@pytest.mark.gpu
def test_a_nan_reaches_the_sums(env):
    """One planted NaN is counted once by the step that reads it, and spreads."""
    _, lbm = env
    cfg, arr = W.random_state(40, 40, seed=2)
    arr = {k: v.copy() for k, v in arr.items()}
    arr["mask"][20, 20] = 0
    arr["T"][20, 20] = np.nan
    s = lbm.Solver(cfg, precision="fp64", diag_every=1).set_geometry(arr).step(1)
    assert s.diagnostics(compute=False)["nonfinite"] == 1
    assert s.step(1).diagnostics(compute=False)["nonfinite"] >= 5
    s.close()


@pytest.mark.gpu
@pytest.mark.parametrize("nx,ny", [(40, 33), (70, 12)])
@pytest.mark.parametrize("every", [1, 5, 12, 50])
def test_coupled_adjoint_with_all_states_equals_checkpoints(env, nx, ny, every, monkeypatch):
    """Keeping every state or recomputing segments from checkpoints (the last
    one short, of one state, or the only one): the same value, gradient, field
    gradient and final state, bit for bit; and a second call goes on from it."""
    _, lbm = env
    cfg, arr = W.random_state(nx, ny, seed=3)
    a = lbm.Solver(cfg, precision="fp64").set_geometry(arr)
    b = lbm.Solver(cfg, precision="fp64").set_geometry(arr)
    va, ga, ta = a.adjoint_coupled(23, observable=0, every=every, initial_T=True)
    monkeypatch.setenv("LBM_ADJOINT_KEEP", "0")
    vb, gb, tb = b.adjoint_coupled(23, observable=0, every=every, initial_T=True)
    assert va == vb and ga == gb and np.array_equal(ta, tb)
    assert a.adjoint_coupled(9, observable=1, axis=1, index=nx // 2, every=every) == \
        b.adjoint_coupled(9, observable=1, axis=1, index=nx // 2, every=4) or \
        np.isnan(a.crossings(1, nx // 2)[0])
    assert a.steps_done == b.steps_done == 32
    fa, fb = a.fields(), b.fields()
    for k in FIELDS:
        assert np.array_equal(fa[k], fb[k]), k
    a.close()
    b.close()


@pytest.mark.gpu
@pytest.mark.parametrize("nx,ny", [(70, 12), (130, 5), (40, 33)])
@pytest.mark.parametrize("diag_every", [1, 3])
def test_coupled_adjoint_steps_as_lbm_step_with_sums(env, nx, ny, diag_every, monkeypatch):
    """A context that reduces its sums every few steps (a column's kernels round
    such steps differently): kept or recomputed states give one value, gradient
    and final state, and that state is lbm_step's, bit for bit."""
    _, lbm = env
    cfg, arr = W.random_state(nx, ny, seed=3)
    a, b, c = (lbm.Solver(cfg, precision="fp64", diag_every=diag_every).set_geometry(arr)
               for _ in range(3))
    va, ga, ta = a.adjoint_coupled(23, observable=0, every=5, initial_T=True)
    monkeypatch.setenv("LBM_ADJOINT_KEEP", "0")
    vb, gb, tb = b.adjoint_coupled(23, observable=0, every=5, initial_T=True)
    assert va == vb and ga == gb and np.array_equal(ta, tb)
    fa, fb, fc = a.fields(), b.fields(), c.step(23).fields()
    for k in FIELDS:
        assert np.array_equal(fa[k], fb[k]) and np.array_equal(fa[k], fc[k]), k
    for s in (a, b, c):
        s.close()


@pytest.mark.gpu
@pytest.mark.parametrize("prec", ["fp32", "fp64"])
def test_batches_of_columns_and_other_grids(env, prec):
    """The two groups advance side by side: however the steps are grouped into
    calls, captured or not, on whichever stream, every context has the same
    fields and sums, bit for bit, and work queued after the call sees them."""
    import torch
    _, lbm = env
    wls = [W.random_state(nx, ny, seed=i)
           for i, (nx, ny) in enumerate([(512, 8), (40, 33), (130, 5), (96, 70), (64, 2)])]

    def solvers():
        return [lbm.Solver(c, precision=prec, diag_every=4).set_geometry(a) for c, a in wls]

    sets = [solvers() for _ in range(3)]
    torch.cuda.synchronize()
    b = lbm.Batch(sets[0])
    b.step(100)
    b.step(23)
    one = lbm.Batch(sets[1])
    for _ in range(123):
        one.step(1)
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        lbm.Batch(sets[2]).step(60).step(63)
        got2 = [s.fields() for s in sets[2]]
    got = [[s.fields() for s in ss] for ss in sets[:2]] + [got2]
    sums = [[s.diagnostics(compute=False) for s in ss] for ss in sets]
    for i in range(len(wls)):
        for k in FIELDS:
            assert np.array_equal(got[0][i][k], got[1][i][k]), (i, k)
            assert np.array_equal(got[0][i][k], got[2][i][k]), (i, k)
        assert sums[0][i] == sums[1][i] == sums[2][i]
    for h in (b, one):
        h.close()
    for ss in sets:
        for s in ss:
            s.close()


@pytest.mark.gpu
@pytest.mark.parametrize("nx,ny,steps,seed", [(144, 100, 25, 7), (222, 175, 19, 33)])
def test_coupled_adjoint_takes_the_fused_form_s_branches(env, nx, ny, steps, seed, monkeypatch):
    """In the gas beside a solid phi = -(1 - phi0) to the last bit, where an ulp
    decides whether the clamp of w passes a derivative.  The gradient on the node
    step's states is that on the fused tile's (form 4): differences of rounding
    alone are of order 1e-14, a branch taken otherwise is 1e-9 in d/dg_y."""
    _, lbm = env
    cfg, arr = W.sessile_droplet(nx, seed=seed, radius=0.2 * min(nx, ny), ny=ny)
    grads = []
    for form in ("0", "4"):
        monkeypatch.setenv("LBM_KERNEL_FORM", form)
        s = lbm.Solver(cfg, precision="fp64").set_geometry(arr)
        grads.append(np.array(s.adjoint_coupled(steps, observable=0, every=16)[1]))
        s.close()
    a, b = grads
    scale = np.abs(b).max()
    assert np.all(np.abs(a - b) <= 1e-11 * np.abs(b) + 1e-13 * scale), (a, b)


@pytest.mark.gpu
@pytest.mark.parametrize("nx,ny", [(70, 12), (40, 33)])
def test_coupled_adjoint_runs_where_the_local_planes_do_not_fit(env, nx, ny, monkeypatch):
    """Memory for the states alone is enough: an allocation with room for their
    local planes that fails is followed by one without, and the results are the
    same, bit for bit."""
    _, lbm = env
    cfg, arr = W.random_state(nx, ny, seed=4)
    monkeypatch.setenv("LBM_ADJOINT_KEEP", "0")
    a, b = (lbm.Solver(cfg, precision="fp64").set_geometry(arr) for _ in range(2))
    va, ga, ta = a.adjoint_coupled(17, observable=0, every=5, initial_T=True)
    lbm.lbm_debug_fail_allocation(0)
    try:
        vb, gb, tb = b.adjoint_coupled(17, observable=0, every=5, initial_T=True)
        c = lbm.Solver(cfg, precision="fp64")  # the hook has fired: this one succeeds
    finally:
        lbm.lbm_debug_fail_allocation(-1)
    assert va == vb and ga == gb and np.array_equal(ta, tb)
    fa, fb = a.fields(), b.fields()
    assert all(np.array_equal(fa[k], fb[k]) for k in FIELDS)
    for s in (a, b, c):
        s.close()


@pytest.mark.gpu
@pytest.mark.parametrize("prec", ["fp64", "tangent", "fp32", "fp16s"])
def test_device_read_outs_are_complete_on_return(env, prec):
    """Fields read into device memory can be taken on any stream, in every
    precision: the call waits for the steps before it and for the read-out."""
    import torch
    _, lbm = env
    cfg, arr = W.random_state(300, 200, seed=1)
    s = lbm.Solver(cfg, precision=prec, tangent={"T_cold": 1.0} if prec == "tangent" else None)
    s.set_geometry(arr).step(64)
    torch.cuda.synchronize()
    out = torch.empty((12, 200, 300), dtype=torch.float64, device="cuda")
    ptrs = [out[k].data_ptr() for k in range(12)]
    s.step(1024)
    lbm.lbm_read_fields(s.ctx, 0xfff, ptrs, lbm.LBM_DEVICE, lbm._stream())
    assert torch.cuda.current_stream().query()
    s.close()


@pytest.mark.gpu
@pytest.mark.parametrize("nx,ny", [(130, 5), (53, 33)])
def test_step_kernel_variable_selects_a_double_form(env, nx, ny, monkeypatch):
    """LBM_STEP_KERNEL=split is the node step on columns too, =fused one kernel a
    step on every grid: the states of the forms that the header names, bit for
    bit, which on this state differ from the other kind's; all match the oracle."""
    O, lbm = env
    cfg, arr = W.random_state(nx, ny, seed=3)
    ref = O.from_workload((cfg, arr)).step(40).fields()

    def run(**env_vars):
        for k, v in env_vars.items():
            monkeypatch.setenv(k, v)
        s = lbm.Solver(cfg, precision="fp64").set_geometry(arr)
        for k in env_vars:
            monkeypatch.delenv(k)
        got = s.step(40).fields()
        s.close()
        _close(got, ref)
        return got

    def same(a, b):
        return all(np.array_equal(a[k], b[k]) for k in FIELDS)

    split, fused = run(LBM_STEP_KERNEL="split"), run(LBM_STEP_KERNEL="fused")
    assert same(split, run(LBM_KERNEL_FORM="1"))
    assert same(fused, run(LBM_KERNEL_FORM="0" if ny < 32 else "4"))
    assert not same(split, fused)


@pytest.mark.gpu
@pytest.mark.parametrize("nx,ny,nz", [(31, 4, 3), (32, 4, 2), (33, 5, 4), (64, 2, 3), (5, 43, 6)])
@pytest.mark.parametrize("seed", [0, 3])
def test_three_dimensional_sizes_match_the_oracle(env, nx, ny, nz, seed):
    """Grids around the float kernels' 32 x 4 x 2 blocks and the double ones'
    128 linear nodes: FP64 at its parity bar, FP32 at 1e-4 in relative L2 (or
    1e-6 of the field's scale), device and host read-outs alike."""
    import torch
    from oracle import oracle3d as O3
    _, lbm = env
    O3.build()
    cfg, arr = W.random_state3(nx, ny, nz, seed=seed)
    ref = O3.from_workload((cfg, arr)).step(15).fields()
    for prec in ("fp64", "fp32"):
        s = lbm.Solver3(cfg, prec).set_geometry(arr).step(15)
        got = s.fields()
        out = torch.full((13, nz, ny, nx), -7.0, dtype=torch.float64, device="cuda")
        lbm.lbm3_read_fields(s.ctx, 0b1010000000101, [out[k].data_ptr() for k in range(13)],
                             lbm.LBM_DEVICE, lbm._stream())
        for i, k in enumerate(lbm.FIELDS3):
            a, b = ref[k], got[k]
            scale = max(np.abs(a).max(), 1e-30)
            if prec == "fp64":
                assert np.abs(a - b).max() <= 1e-10 * scale, k
            else:
                den = max(np.linalg.norm(a), 1e-30 * np.sqrt(a.size))
                assert np.linalg.norm(a - b) <= 1e-4 * den or \
                    np.abs(a - b).max() <= 1e-6 * max(scale, 1e-3), k
            want = b if 0b1010000000101 >> i & 1 else np.full_like(b, -7.0)
            assert np.array_equal(out[i].cpu().numpy(), want), k
        s.close()


def _fma(a, b, c):
    return float(Fraction(a) * Fraction(b) + Fraction(c))  # one rounding, as the device's fma


def test_third_order_reciprocal_is_within_an_ulp():
    """r = r0 + r0 (e + e^2), e = 1 - b r0, from any seed within 2^-19 of 1 / b
    (the hardware's approximation is nearer): less than one ulp off; and the
    quotient corrected by its residual likewise."""
    r = np.random.default_rng(5)
    for _ in range(2000):
        b = float(2.0 ** r.uniform(-30, 30))
        r0 = float(Fraction(1) / Fraction(b) * (1 + Fraction(float(r.uniform(-1, 1)) * 2.0 ** -19)))
        e = _fma(-b, r0, 1.0)
        x = _fma(r0, _fma(e, e, e), r0)
        exact = Fraction(1) / Fraction(b)
        assert abs(Fraction(x) - exact) < Fraction(float(np.spacing(float(exact))))
        a = float(r.uniform(-3, 3))
        q0 = a * x
        q = _fma(_fma(-q0, b, a), x, q0)
        exact = Fraction(a) / Fraction(b)
        assert abs(Fraction(q) - exact) < Fraction(float(np.spacing(abs(float(exact)))))


PROBE = r"""
#include "lbm_node.cuh"
__global__ void probe(const double* a, const double* b, double* r, double* q, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  r[i] = lbmn::rcp(b[i]);
  q[i] = lbmn::quot(a[i], b[i]);
}
extern "C" int run_probe(const double* a, const double* b, double* r, double* q, int n) {
  probe<<<(n + 255) / 256, 256>>>(a, b, r, q, n);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.mark.gpu
def test_device_reciprocal_and_quotient_are_within_an_ulp(env, tmp_path):
    """rcp and quot of lbm_node.cuh on the device, hardware seed and all, against
    the IEEE results: mantissas at and beside the powers of two, and random ones,
    over exponents whose reciprocals and quotients are normal numbers."""
    import ctypes
    import subprocess

    import torch
    from paper_2510_18688_gb300 import build
    (tmp_path / "probe.cu").write_text(PROBE)
    so = tmp_path / "probe.so"
    subprocess.run([build.nvcc(), build.ARCH, "-O3", "-std=c++17", "-Xcompiler", "-fPIC", "-shared",
                    "-I", build.SRC, str(tmp_path / "probe.cu"), "-o", str(so)], check=True)
    r = np.random.default_rng(11)
    n = 1 << 21
    m = np.concatenate([r.uniform(1.0, 2.0, n), 1.0 + np.arange(4096) * 2.0 ** -52,
                        2.0 - np.arange(1, 4097) * 2.0 ** -52, 1.0 + np.arange(8192) / 8192.0])
    b = np.ldexp(m, r.integers(-500, 501, m.size))
    a = np.ldexp(r.permutation(m), r.integers(-500, 501, m.size)) * r.choice([-1.0, 1.0], m.size)
    ta, tb = (torch.as_tensor(v, device="cuda") for v in (a, b))
    tr, tq = torch.empty_like(tb), torch.empty_like(tb)
    torch.cuda.synchronize()
    f = ctypes.CDLL(str(so)).run_probe
    f.argtypes = [ctypes.c_void_p] * 4 + [ctypes.c_int]
    assert f(ta.data_ptr(), tb.data_ptr(), tr.data_ptr(), tq.data_ptr(), m.size) == 0
    for got, want in ((tr.cpu().numpy(), 1.0 / b), (tq.cpu().numpy(), a / b)):
        assert np.all(np.abs(got - want) <= np.spacing(np.abs(want)))
