"""What the complex128 sweeps in digits and of small spaces must leave as the FP64
engine (FS_SWEEP_CUDA_CORE) has it: programs and amplitudes that are not
numbers, and vectors whose amplitudes span many orders of magnitude.

The FP64 form inside the digit sweep applies the same rotations in the same
order to every amplitude as that engine, so that they differ by the rounding of
the phases behind each spin's rotations: a few 2^-53 of an amplitude after the
first spin, which the second spin's rotations carry to at most a few hundred
2^-53 = 1e-13 of the largest amplitude that they mix it with (TOL)."""

import os

import numpy as np
import pytest

from paper_2605_03123_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-13


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


def _both(lib, ctx, f, engine="FS_SWEEP_TENSOR"):
    """f() under the digit engine and under the FP64 one, and the first's kernels."""
    ctx.set_sweep_engine(getattr(lib, engine))
    ctx.profile_start()
    got = f()
    used = ctx.profile_stop()
    assert ctx.sync_status() == 0
    ctx.set_sweep_engine(lib.FS_SWEEP_CUDA_CORE)
    return got, f(), used


@pytest.mark.parametrize("engine", ["FS_SWEEP_AUTO", "FS_SWEEP_TENSOR"])
@pytest.mark.parametrize("norb,nelec", [(6, (3, 3)), (8, (4, 4)), (12, (6, 5))])
@pytest.mark.parametrize("where", ["diagonal", "row", "all"])
def test_rotation_that_is_not_a_number(lib, ctx, norb, nelec, where, engine):
    """A NaN in U reaches the amplitudes that it reaches in FP64 (it passes the
    unitarity check, whose maximum ignores it): from the first diagonal entry
    only the diagonal layer, from others the rotations too."""
    g = inputs.rng(42100 + norb)
    U = inputs.haar_unitary(norb, g)
    if where == "diagonal":
        U[0, 0] = np.nan
    elif where == "row":
        U[norb // 2] = np.nan
    else:
        U[:] = np.nan
    v = inputs.random_state(norb, nelec, g)
    got, ref, _ = _both(lib, ctx, lambda: lib.apply_orbital_rotation_(
        torch.from_numpy(v).cuda(), U, norb, nelec, ctx=ctx).cpu().numpy(), engine)
    assert np.isnan(ref).any()
    assert (np.isnan(got) == np.isnan(ref)).all()


def _block_diagonal(norb, g):
    U = np.zeros((norb, norb), complex)
    h = norb // 2
    U[:h, :h] = inputs.haar_unitary(h, g)
    U[h:, h:] = inputs.haar_unitary(norb - h, g)
    return U


def _levels(lib, ctx, norb, nelec, mask):
    """Per spin, the electrons of every string outside the orbitals in mask."""
    return [np.array([bin(int(m) & ~mask).count("1") for m in lib.string_table(norb, n, ctx=ctx)])
            for n in nelec]


def _close_by_level(got, ref, la, lb):
    """Every block of one level of each spin to TOL of its own largest amplitude."""
    for a in np.unique(la):
        for b in np.unique(lb):
            at = np.ix_(la == a, lb == b)
            scale = np.max(np.abs(ref[at]))
            assert np.max(np.abs(got[at] - ref[at])) <= TOL * scale, (a, b, scale)


# one and many vectors a slab, both spins, slabs with both kinds of vectors
RANGE_SECTORS = [(8, (4, 3)), (10, (5, 5)), (11, (3, 8)), (12, (6, 2)), (13, (6, 1)), (12, (6, 6))]


@pytest.mark.parametrize("norb,nelec", RANGE_SECTORS)
@pytest.mark.parametrize("step", [1e-7, 1e-4])
def test_small_blocks_of_a_block_diagonal_rotation(lib, ctx, norb, nelec, step):
    """A rotation that keeps the electrons of each half of the orbitals: blocks
    of `step` to the power of the electrons in the upper half, down to 1e-84
    of the state, keep their own accuracy."""
    g = inputs.rng(42200 + 31 * norb + nelec[0])
    U = _block_diagonal(norb, g)
    la, lb = _levels(lib, ctx, norb, nelec, (1 << (norb // 2)) - 1)
    v = inputs.random_state(norb, nelec, g)
    v *= step ** (la[:, None] + lb[None, :]).astype(float)
    got, ref, used = _both(lib, ctx, lambda: lib.apply_orbital_rotation_(
        torch.from_numpy(v).cuda(), U, norb, nelec, ctx=ctx).cpu().numpy())
    assert any(k.endswith("_fx") for k in used), used
    _close_by_level(got, ref, la, lb)


@pytest.mark.parametrize("norb,nelec", [(8, (4, 3)), (10, (1, 5)), (11, (2, 4)), (12, (2, 3))])
@pytest.mark.parametrize("kind", ["weak", "weaker", "blocks"])
def test_vectors_that_start_with_zeros(lib, ctx, norb, nelec, kind):
    """One spin rotated, against the sweep of small spaces, which applies the
    rotations in the same order (the window sweeps reorder commuting ones), so
    that the two may differ in the product with the phase alone: 8 2^-53 in
    the modulus of an amplitude, in its angle what the reference's angles are
    good to (TOL).  Determinants whose excitations come out tiny (below 2^-32
    of the vector, a factor of four inside the rule), among spread vectors and
    zero ones."""
    import scipy.linalg
    g = inputs.rng(42300 + 31 * norb + nelec[0])
    if kind == "blocks":  # joined by one rotation of 1e-7
        R = np.eye(norb)
        k = norb // 2
        R[k - 1:k + 1, k - 1:k + 1] = [[np.cos(1e-7), np.sin(1e-7)], [-np.sin(1e-7), np.cos(1e-7)]]
        U = _block_diagonal(norb, g) @ R
    else:
        U = scipy.linalg.expm(inputs.random_antihermitian(norb, 3e-3 if kind == "weak" else 3e-5, g))
    I = np.eye(norb)
    v = inputs.random_state(norb, nelec, g)
    rows = np.arange(v.shape[0]) % 4
    one = np.zeros_like(v)
    one[np.arange(v.shape[0]), g.integers(0, v.shape[1], v.shape[0])] = 1e-3
    v = np.where((rows == 0)[:, None], v, np.where((rows == 1)[:, None], 0, one))

    def both(f, spin):
        out = []
        for engine, kernel in ((lib.FS_SWEEP_TENSOR, "fx"), (lib.FS_SWEEP_AUTO, "pairs")):
            ctx.set_sweep_engine(engine)
            ctx.profile_start()
            out.append(f().cpu().numpy())
            used = ctx.profile_stop()
            assert "sweep_%s_%s" % (spin, kernel) in used, used
        return out
    got, ref = both(lambda: lib.apply_orbital_rotation_(
        torch.from_numpy(v).cuda(), I, norb, nelec, U_b=U, ctx=ctx), "beta")
    norm = np.linalg.norm(ref, axis=1, keepdims=True)
    small = np.where(ref == 0, np.inf, np.abs(ref)).min(1, keepdims=True) < 2.0 ** -32 * norm

    def check(got, ref):
        assert (np.abs(got - ref) <= TOL * np.where(small, np.abs(ref), norm)).all()
        moduli = np.abs(np.abs(got) - np.abs(ref))
        assert (moduli <= np.where(small, 8 * 2.0 ** -53 * np.abs(ref), TOL * norm)).all()
    check(got, ref)
    assert small[rows > 1].any() or kind != "weaker"
    # the other spin: columns
    got, ref = both(lambda: lib.apply_orbital_rotation_(
        torch.from_numpy(v.T.copy()).cuda(), U, norb, nelec[::-1], U_b=I, ctx=ctx).T, "alpha")
    check(got, ref)


@pytest.mark.parametrize("norb,nelec", [(8, (4, 3)), (12, (6, 2)), (12, (5, 6))])
def test_amplitudes_that_are_not_numbers_stay_in_their_block(lib, ctx, norb, nelec):
    """Infinities and NaNs reach the amplitudes that they reach in FP64."""
    g = inputs.rng(42400 + norb)
    U = _block_diagonal(norb, g)
    v = inputs.random_state(norb, nelec, g)
    v[1, 2] = np.nan
    v[3, 0] = np.inf
    v[-1, -1] = complex(0, -np.inf)
    got, ref, _ = _both(lib, ctx, lambda: lib.apply_orbital_rotation_(
        torch.from_numpy(v).cuda(), U, norb, nelec, ctx=ctx).cpu().numpy())
    ok = np.isfinite(ref)
    assert ok.any() and not ok.all()
    assert (np.isfinite(got) == ok).all()
    assert np.max(np.abs(got[ok] - ref[ok])) <= TOL


def test_phases_behind_a_rotation_of_wide_range(lib, ctx):
    """The diagonal gate fused behind the rotation (cross tables and string
    phases) on vectors of both kinds, with a coupling that is not a number."""
    norb, nelec = 12, (6, 2)
    g = inputs.rng(42500)
    U = _block_diagonal(norb, g)[None]
    J = inputs.random_symmetric(norb, 1.0, g)[None]
    h = np.diag(g.normal(0, 1, norb)).astype(complex)
    la, lb = _levels(lib, ctx, norb, nelec, (1 << (norb // 2)) - 1)
    v = inputs.random_state(norb, nelec, g)
    v *= 1e-6 ** (la[:, None] + lb[None, :]).astype(float)
    run = lambda: lib.simulate_trotter_double_factorized_(
        torch.from_numpy(v).cuda(), h, J, U, 0.4, norb, nelec, ctx=ctx).cpu().numpy()
    got, ref, used = _both(lib, ctx, run)
    assert any(k.endswith("_fx") for k in used), used
    _close_by_level(got, ref, la, lb)
    J[0, 2, 9] = J[0, 9, 2] = np.inf
    got, ref, _ = _both(lib, ctx, run)
    assert np.isnan(ref).any() and (np.isnan(got) == np.isnan(ref)).all()


@pytest.mark.parametrize("norb,nelec", [(8, (4, 4)), (10, (5, 4)), (12, (6, 5))])
@pytest.mark.parametrize("swap", [False, True])
def test_gradient_entries_between_blocks(lib, ctx, norb, nelec, swap):
    """Generators that keep each half of the orbitals, a state and a cotangent
    whose blocks (electrons in the upper half) step down by 1e-9, or one up
    and one down: the entries of dK between the halves, 1e-9 of the others and
    less, to TOL of the largest of them.  (Each is a sum over the amplitudes
    that the excitation joins, where FP64 rounds at 2^-53 of these.)"""
    g = inputs.rng(42600 + norb)
    h = norb // 2
    K = np.zeros((2, norb, norb), complex)
    for k in K:
        k[:h, :h] = inputs.random_antihermitian(h, 0.5, g)
        k[h:, h:] = inputs.random_antihermitian(norb - h, 0.5, g)
    Ja = np.array([inputs.random_symmetric(norb, 0.5, g) for _ in range(2)])
    Jb = np.array([inputs.random_symmetric(norb, 0.5, g) for _ in range(2)])
    la, lb = _levels(lib, ctx, norb, nelec, (1 << h) - 1)
    level = (la[:, None] + lb[None, :]).astype(float)
    v, cot = inputs.random_state(norb, nelec, g), inputs.random_state(norb, nelec, g)
    v *= 1e-9 ** level
    cot *= 1e-9 ** (level.max() - level if swap else level)

    def run():
        x, c = torch.from_numpy(v).cuda(), torch.from_numpy(cot).cuda()
        lib.lucj_forward_(x, K, Ja, Jb, norb, nelec, ctx=ctx)
        dK = lib.lucj_vjp_(x, c, K, Ja, Jb, norb, nelec, ctx=ctx)[0]
        return dK, c.cpu().numpy()
    got, ref, used = _both(lib, ctx, run)
    assert any(k.startswith("trans_") for k in used), used
    for block in (np.s_[:, :h, :h], np.s_[:, h:, h:], np.s_[:, :h, h:], np.s_[:, h:, :h]):
        scale = np.max(np.abs(ref[0][block]))
        assert scale > 0
        assert np.max(np.abs(got[0][block] - ref[0][block])) <= TOL * scale, (block, scale)
    _close_by_level(got[1], ref[1], la, lb)


def test_rotation_method_is_measured_per_engine(lib):
    """FS_ROT_AUTO times sweeps and minors once under each sweep engine: the
    sweeps of another engine take another time."""
    c = lib.Context(0)
    norb, nelec = 9, (4, 5)
    g = inputs.rng(42800)
    U = inputs.haar_unitary(norb, g)
    x = torch.from_numpy(inputs.random_state(norb, nelec, g)).cuda()
    measured = []
    for engine in (lib.FS_SWEEP_CUDA_CORE, lib.FS_SWEEP_AUTO, lib.FS_SWEEP_CUDA_CORE):
        c.set_sweep_engine(engine)
        c.profile_start()
        lib.apply_orbital_rotation_(x, U, norb, nelec, ctx=c)
        used = c.profile_stop()
        measured.append(any(k.startswith("minor_") for k in used)
                        and any(k.startswith("sweep_") for k in used))
    c.close()
    assert measured == [True, True, False]


@pytest.mark.parametrize("norb,nelec,gate,kernel", [
    (12, (12, 6), "dense", "sweep_beta_fx"), (12, (12, 6), "givens", "sweep_beta_f64"),
    (13, (0, 4), "block", "sweep_beta_f64"), (13, (2, 7), "block", "sweep_beta_fx"),
    (14, (1, 4), "block", "sweep_beta_f64"), (14, (4, 4), "block", "sweep_beta_fx")])
def test_small_programs_on_few_vectors_stay_in_fp64(lib, ctx, norb, nelec, gate, kernel):
    """Where the digit sweep's images and steps take longer than the rotations."""
    g = inputs.rng(42900 + norb)
    U = inputs.haar_unitary(norb, g)
    if gate == "givens":
        c, s = np.cos(0.3), np.sin(0.3)
        U = np.eye(norb)
        U[np.ix_([0, norb - 1], [0, norb - 1])] = [[c, s], [-s, c]]
    elif gate == "block":
        h = norb // 2
        U = np.eye(norb, dtype=complex)
        U[:h, :h] = inputs.haar_unitary(h, g)
    v = torch.from_numpy(inputs.random_state(norb, nelec, g)).cuda()
    got, ref, used = _both(lib, ctx, lambda: lib.apply_orbital_rotation(
        v, np.eye(norb), norb, nelec, U_b=U, ctx=ctx), "FS_SWEEP_AUTO")
    assert kernel in used, used
    assert float((got - ref).abs().max()) <= TOL


def test_without_room_for_the_images(lib, ctx):
    """A call whose images cannot be allocated rotates in FP64."""
    norb, nelec = 12, (6, 6)
    g = inputs.rng(43000)
    U = inputs.haar_unitary(norb, g)
    v = torch.from_numpy(inputs.random_state(norb, nelec, g)).cuda()
    x = v.clone()
    ctx.set_sweep_engine(lib.FS_SWEEP_CUDA_CORE)
    ref = lib.apply_orbital_rotation(v, U, norb, nelec, ctx=ctx)
    ctx.set_sweep_engine(lib.FS_SWEEP_AUTO)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    hold = []
    try:
        for left in (256, 32, 4):  # MB; the images take 8.8
            free = torch.cuda.mem_get_info()[0] - (left << 20)
            if free > 0:
                hold.append(torch.empty(free, dtype=torch.uint8, device="cuda"))
        ctx.profile_start()
        lib.apply_orbital_rotation_(x, U, norb, nelec, ctx=ctx)
        used = ctx.profile_stop()
    finally:
        hold.clear()
        torch.cuda.empty_cache()
    assert not any(k.endswith("_fx") for k in used), used
    assert torch.equal(x, ref)
    lib.apply_orbital_rotation_(x, U, norb, nelec, ctx=ctx)  # with room again
    assert ctx.sync_status() == 0
