"""What the complex128 sweeps in digits and of small spaces must leave as the FP64
engine (FS_SWEEP_CUDA_CORE) has it."""

import os

import numpy as np
import pytest

from paper_2605_03123_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


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
