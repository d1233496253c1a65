"""Calls inside a stream capture after a warm call of the same kind with other
arguments: nothing that the sector or the type decides may be left to
allocate."""

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


def _captured(f):
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        out = f()
    graph.replay()
    torch.cuda.synchronize()
    return out


def _programs(norb, g):
    dense = inputs.haar_unitary(norb, g)
    block = np.eye(norb, dtype=complex)
    block[:4, :4] = inputs.haar_unitary(4, g)
    gate = np.eye(norb, dtype=complex)
    gate[1:3, 1:3] = inputs.haar_unitary(2, g)
    return dense, block, gate


@pytest.mark.parametrize("dt", [torch.complex64, torch.complex128])
@pytest.mark.parametrize("norb,nelec", [(8, (4, 4)), (10, (5, 5)), (12, (6, 4))])
@pytest.mark.parametrize("warm,then", [(0, 1), (1, 0), (2, 0), (0, 2)])
def test_rotations_after_a_warm_call_of_another_program(lib, ctx, dt, norb, nelec, warm, then):
    """Dense, within four orbitals, and a single gate: the sweeps that take them
    differ."""
    g = inputs.rng(43000 + norb)
    U = _programs(norb, g)
    v = torch.from_numpy(inputs.random_state(norb, nelec, g)).cuda().to(dt)
    x = v.clone()
    lib.apply_orbital_rotation_(x, U[warm], norb, nelec, ctx=ctx)
    torch.cuda.synchronize()
    x.copy_(v)
    _captured(lambda: lib.apply_orbital_rotation_(x, U[then], norb, nelec, ctx=ctx))
    ref = lib.apply_orbital_rotation(v, U[then], norb, nelec, ctx=ctx)
    assert torch.equal(x, ref)


@pytest.mark.parametrize("dt", [torch.complex64, torch.complex128])
def test_more_shots_than_the_warm_call(lib, ctx, dt):
    norb, nelec = 9, (4, 5)
    g = inputs.rng(43100)
    v = torch.from_numpy(inputs.random_state(norb, nelec, g)).cuda().to(dt)
    u = torch.from_numpy(g.random(200000)).cuda()
    lib.sample_state(v, norb, nelec, uniforms=u[:10], ctx=ctx)
    torch.cuda.synchronize()
    got = _captured(lambda: lib.sample_state(v, norb, nelec, uniforms=u, ctx=ctx))
    assert torch.equal(got, lib.sample_state(v, norb, nelec, uniforms=u, ctx=ctx))


def test_digit_sweep_of_a_space_known_to_fp64_only(lib, ctx):
    """A captured call under FS_SWEEP_AUTO after warm ones under the FP64 engine."""
    norb, nelec = 12, (6, 5)
    g = inputs.rng(43200)
    U = inputs.haar_unitary(norb, g)
    v = torch.from_numpy(inputs.random_state(norb, nelec, g)).cuda()
    ctx.set_sweep_engine(lib.FS_SWEEP_CUDA_CORE)
    ref = lib.apply_orbital_rotation(v, U, norb, nelec, ctx=ctx)
    ctx.set_sweep_engine(lib.FS_SWEEP_AUTO)
    x = v.clone()
    torch.cuda.synchronize()
    _captured(lambda: lib.apply_orbital_rotation_(x, U, norb, nelec, ctx=ctx))
    assert torch.equal(x, ref)
