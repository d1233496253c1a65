"""The complex128 orbital rotation on the tensor cores (fixed-point digits)
against the oracle and against the FP64 sweeps.  The tolerance is the library's
for complex128 amplitudes, 1e-12 of a unit-norm state: each of up to a dozen
window steps rounds an amplitude at 2^-60 of its vector's norm."""

import os

import numpy as np
import pytest

import oracle
from paper_2605_03123_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-12


@pytest.fixture(scope="module", autouse=True)
def lib():
    assert torch.cuda.is_available(), "the GPU tests need a CUDA device"
    from paper_2605_03123_gb300 import build, fsgpu
    if not os.path.exists(build.lib_path()):
        build.build()
    fsgpu.load_library()
    return fsgpu


@pytest.fixture
def ctx(lib):
    c = lib.Context(0)
    c.set_rotation_path(lib.FS_ROT_GIVENS)
    yield c
    c.close()


def _kernels(ctx, f):
    ctx.profile_start()
    f()
    return ctx.profile_stop()


# every window class (m = 1 .. 6) alone and together, steps without class 3,
# one row, ragged tiles, rows past a tile, many and single vectors per slab
SECTORS = [(6, (3, 4)), (7, (2, 5)), (8, (1, 7)), (8, (4, 6)), (9, (8, 4)), (10, (5, 5)),
           (11, (9, 3)), (12, (6, 2)), (13, (6, 1)), (16, (3, 2)), (20, (2, 2))]


@pytest.mark.parametrize("norb,nelec", SECTORS)
def test_against_oracle_and_fp64_sweeps(lib, ctx, norb, nelec):
    g = inputs.rng(41000 + 37 * norb + 5 * nelec[0] + nelec[1])
    Ua, Ub = inputs.haar_unitary(norb, g), inputs.haar_unitary(norb, g)
    v = inputs.random_state(norb, nelec, g)
    ref = oracle.apply_orbital_rotation(v, Ua, Ub, norb, nelec)
    x = torch.from_numpy(v).cuda()
    y = x.clone()
    ctx.set_sweep_engine(lib.FS_SWEEP_TENSOR)
    used = _kernels(ctx, lambda: lib.apply_orbital_rotation_(x, Ua, norb, nelec, U_b=Ub, ctx=ctx))
    assert ctx.sync_status() == 0
    assert v.size < 400 or any(k.endswith("_fx") for k in used), used
    assert np.max(np.abs(x.cpu().numpy() - ref)) < TOL
    ctx.set_sweep_engine(lib.FS_SWEEP_CUDA_CORE)
    used = _kernels(ctx, lambda: lib.apply_orbital_rotation_(y, Ua, norb, nelec, U_b=Ub, ctx=ctx))
    assert not any(k.endswith("_fx") for k in used), used
    assert float((x - y).abs().max()) < TOL


@pytest.mark.parametrize("engine", ["FS_SWEEP_AUTO", "FS_SWEEP_TENSOR"])
@pytest.mark.parametrize("scale", [1e-305, 1e-150, 1e150])
def test_scales_and_zero_vectors(lib, ctx, scale, engine):
    """Each vector keeps its own scale: rows of very different size (and zero
    rows and columns) come out as accurate as a rotation of each alone."""
    ctx.set_sweep_engine(getattr(lib, engine))
    norb, nelec = 9, (4, 5)
    g = inputs.rng(41900)
    U = inputs.haar_unitary(norb, g)
    I = np.eye(norb)
    v = inputs.random_state(norb, nelec, g)
    rows = 10.0 ** -np.arange(v.shape[0]).clip(0, 100)
    rows[3] = 0.0
    ref = oracle.apply_orbital_rotation(v, I, U, norb, nelec) * rows[:, None]
    x = torch.from_numpy(v * rows[:, None] * scale).cuda()
    lib.apply_orbital_rotation_(x, I, norb, nelec, U_b=U, ctx=ctx)
    assert ctx.sync_status() == 0
    out = x.cpu().numpy() / scale
    tiny = 5e-324 / scale * 20  # FP64 subnormal spacing of the scaled values
    err = np.abs(out - ref).max(1)
    assert (err <= 1e-12 * np.abs(ref).max(1) + tiny).all(), err
    assert not out[3].any()


@pytest.mark.parametrize("engine", ["FS_SWEEP_AUTO", "FS_SWEEP_TENSOR"])
def test_not_finite_vectors_stay_apart(lib, ctx, engine):
    ctx.set_sweep_engine(getattr(lib, engine))
    norb, nelec = 8, (4, 4)
    g = inputs.rng(41950)
    U = inputs.haar_unitary(norb, g)
    I = np.eye(norb)
    v = inputs.random_state(norb, nelec, g)
    ref = oracle.apply_orbital_rotation(v, I, U, norb, nelec)
    bad = v.copy()
    bad[5, 17] = np.nan
    bad[40, 0] = np.inf
    x = torch.from_numpy(bad).cuda()
    lib.apply_orbital_rotation_(x, I, norb, nelec, U_b=U, ctx=ctx)
    out = x.cpu().numpy()
    keep = np.ones(v.shape[0], bool)
    keep[[5, 40]] = False
    assert np.max(np.abs(out[keep] - ref[keep])) < TOL
    assert not np.isfinite(out[5]).all() and not np.isfinite(out[40]).all()


def test_single_givens_gate_leaves_other_strings_alone(lib, ctx):
    """A program of few rotations keeps the FP64 sweep: amplitudes it does not
    mix are returned bit for bit."""
    norb, nelec = 10, (5, 5)
    v = inputs.random_state(norb, nelec, inputs.rng(41970))
    x = torch.from_numpy(v).cuda()
    lib.apply_givens_rotation_(x, 0.3, 2, 3, norb, nelec, spin="beta", ctx=ctx)
    m = lib.string_table(norb, 5, ctx=ctx)
    same = ((m >> 2) & 1) == ((m >> 3) & 1)
    assert (x.cpu().numpy()[:, same] == v[:, same]).all()


@pytest.mark.parametrize("norb,nelec", [(7, (3, 3)), (9, (5, 4))])
def test_vjp_against_oracle(lib, ctx, norb, nelec):
    g = inputs.rng(41980 + norb)
    K = np.array([inputs.random_antihermitian(norb, 0.5, g) for _ in range(2)])
    Ja = np.array([inputs.random_symmetric(norb, 0.5, g) for _ in range(2)])
    Jb = np.array([inputs.random_symmetric(norb, 0.5, g) for _ in range(2)])
    v, cot = inputs.random_state(norb, nelec, g), inputs.random_state(norb, nelec, g)
    ref = oracle.lucj_forward(K, Ja, Jb, norb, nelec, vec=v)
    grads = oracle.lucj_vjp(K, Ja, Jb, cot, norb, nelec, vec=v)
    x, c = torch.from_numpy(v).cuda(), torch.from_numpy(cot).cuda()
    lib.lucj_forward_(x, K, Ja, Jb, norb, nelec, ctx=ctx)
    assert np.max(np.abs(x.cpu().numpy() - ref)) < TOL
    got = lib.lucj_vjp_(x, c, K, Ja, Jb, norb, nelec, ctx=ctx)
    assert ctx.sync_status() == 0
    for a, b in zip(got, grads):
        assert np.max(np.abs(a - b)) <= 1e-10 * max(1.0, np.max(np.abs(b)))
    assert np.max(np.abs(c.cpu().numpy() - grads[3])) < TOL
    assert np.max(np.abs(x.cpu().numpy() - v)) < TOL


def test_phase_of_non_finite_coupling_stays_with_its_strings(lib, ctx):
    """The complex128 phase passes: a coupling that is not a number reaches the
    configurations that hold both its orbitals, and no others."""
    norb, nelec = 9, (4, 5)
    g = inputs.rng(41990)
    v = inputs.random_state(norb, nelec, g)
    Ja, Jb = inputs.random_symmetric(norb, 1.0, g), inputs.random_symmetric(norb, 1.0, g)
    ref = oracle.apply_diag_coulomb_evolution(v, Ja, Jb, Ja, 0.4, norb, nelec)
    Jb = Jb.copy()
    Jb[2, 7] = np.nan
    x = torch.from_numpy(v).cuda()
    lib.apply_diag_coulomb_evolution_(x, Ja, Jb, 0.4, norb, nelec, ctx=ctx)
    ma, mb = lib.string_table(norb, 4, ctx=ctx), lib.string_table(norb, 5, ctx=ctx)
    hit = (((ma >> 2) & 1)[:, None] & ((mb >> 7) & 1)[None, :]).astype(bool)
    out = x.cpu().numpy()
    assert np.isnan(out[hit]).all()
    assert np.max(np.abs(out[~hit] - ref[~hit])) < TOL


@pytest.mark.parametrize("norb,nelec", [(2, (1, 1)), (4, (2, 1)), (5, (4, 3)), (8, (4, 4)),
                                        (9, (5, 4)), (9, (1, 8)), (12, (2, 1)), (17, (1, 2))])
def test_small_spaces_against_fp64_window_sweeps(lib, ctx, norb, nelec):
    """The sweep of small spaces applies the same rotations in the same order
    with the same FP64 operations as the window sweeps: only the phases behind
    them round differently.  Also with its own cross tables (a diagonal gate
    fused behind the rotation)."""
    g = inputs.rng(42000 + 41 * norb + nelec[0])
    Ua, Ub = inputs.haar_unitary(norb, g), inputs.haar_unitary(norb, g)
    h, J = inputs.random_symmetric(norb, 0.7, g), inputs.random_symmetric(norb, 0.7, g)
    v = inputs.random_state(norb, nelec, g)
    ref = oracle.apply_orbital_rotation(v, Ua, Ub, norb, nelec)
    tref = oracle.simulate_trotter_diag_coulomb(v, h, J, J, J, 0.6, norb, nelec, 2, 1)
    out = []
    for engine in (lib.FS_SWEEP_AUTO, lib.FS_SWEEP_CUDA_CORE):
        ctx.set_sweep_engine(engine)
        x = torch.from_numpy(v).cuda()
        used = _kernels(ctx, lambda: lib.apply_orbital_rotation_(x, Ua, norb, nelec, U_b=Ub, ctx=ctx))
        # N = 17 has too many rotations for a sweep one rotation at a time
        taken = engine == lib.FS_SWEEP_AUTO and norb <= 12
        assert any("pairs" in k for k in used) == taken, used
        y = torch.from_numpy(v).cuda()
        lib.simulate_trotter_diag_coulomb_(y, h, J, J, 0.6, norb, nelec, n_steps=2, order=1, ctx=ctx)
        assert np.max(np.abs(y.cpu().numpy() - tref)) < TOL
        out.append(x.cpu().numpy())
    assert np.max(np.abs(out[0] - ref)) < TOL
    assert np.max(np.abs(out[0] - out[1])) < 1e-14 * norb
