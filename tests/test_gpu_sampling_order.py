"""Shots ordered by group (calls of MANY shots) against the same uniforms drawn a
FEW at a time, one warp each, where the two could part: slices without mass
inside a group, targets on the rounding of the prefix sums, and states that put
all shots into a few groups."""

import os

import numpy as np
import pytest

from paper_2605_03123_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# above and below the lines of both types for up to 3000 groups of 256 amplitudes
MANY, FEW = 130_000, 9_000


@pytest.fixture(scope="module", autouse=True)
def lib():
    assert torch.cuda.is_available(), "the GPU tests need a CUDA device"
    from paper_2605_03123_gb300 import build, fsgpu
    if not os.path.exists(build.lib_path()):
        build.build()
    fsgpu.load_library()
    return fsgpu


def _sums(p):
    """FP64 sums of one group of 256 masses as the kernels form them: the
    total (each of 32 lanes eight strided masses, then a butterfly), and the
    inclusive shuffle scan over the 32 slices of eight neighbours."""
    lane = np.zeros(32)
    for k in range(8):
        lane = lane + p[32 * k:32 * k + 32]
    for m in (16, 8, 4, 2, 1):
        lane = lane + lane[np.arange(32) ^ m]
    own = np.zeros(32)
    for k in range(8):
        own = own + p[k::8]
    incl = own.copy()
    for d in (1, 2, 4, 8, 16):
        y = incl.copy()
        y[d:] = incl[:-d] + incl[d:]
        incl = y
    return lane[0], own, incl


def _gap_uniforms(x):
    """Uniforms whose target is the sum before an empty slice, where that
    slice's own sum lies above it."""
    total, own, incl = _sums(x * x)
    out = []
    for l in range(1, 31):
        if own[l] == 0 and incl[l] > incl[l - 1] and (own[l + 1:] > 0).sum() > 1:
            u = incl[l - 1] / total
            for w in (u, np.nextafter(u, 0), np.nextafter(u, 1)):
                if w * total == incl[l - 1]:
                    out.append(w)
                    break
    return out


def test_target_in_the_rounding_of_an_empty_slice(lib):
    """The shuffle scan adds in another order per lane, so that a slice without
    mass can end above the one before it: a target between the two belongs to
    the next slice with mass, in both forms of the search."""
    norb, nelec = 6, (3, 3)  # 400 amplitudes: two groups, the second empty
    found = 0
    for seed in range(40):
        g = inputs.rng(1700 + seed)
        x = np.zeros(400)
        x[:256] = g.standard_normal(256) * np.repeat(g.random(32) < 0.6, 8)
        us = _gap_uniforms(x[:256])
        if not us:
            continue
        found += len(us)
        v = torch.from_numpy(x.astype(np.complex128).reshape(20, 20)).cuda()
        alone = lib.sample_state(v, norb, nelec, uniforms=np.array(us))
        u2 = np.concatenate([us, g.random(MANY)])
        got = lib.sample_state(v, norb, nelec, uniforms=u2)[:len(us)]
        assert torch.equal(got, alone), (seed, got, alone)
    assert found > 10


@pytest.mark.parametrize("dt", [torch.complex64, torch.complex128])
@pytest.mark.parametrize("norb,nelec", [(6, (3, 3)), (8, (4, 4)), (12, (6, 5))])
def test_states_with_empty_slices(lib, dt, norb, nelec):
    """Six in ten slices of eight amplitudes empty, single amplitudes too."""
    g = inputs.rng(1750 + norb)
    v = inputs.random_state(norb, nelec, g)
    flat = v.reshape(-1)
    flat[np.repeat(g.random((flat.size + 7) // 8) < 0.6, 8)[:flat.size]] = 0
    flat[g.random(flat.size) < 0.2] = 0
    x = torch.from_numpy(v).cuda().to(dt)
    u = torch.from_numpy(g.random(MANY)).cuda()
    got = lib.sample_state(x, norb, nelec, uniforms=u)
    alone = torch.cat([lib.sample_state(x, norb, nelec, uniforms=u[i:i + FEW])
                       for i in range(0, MANY, FEW)])
    assert torch.equal(got, alone)


@pytest.mark.parametrize("dt", [torch.complex64, torch.complex128])
def test_ends_and_unusable_states(lib, dt):
    """The ends of the uniform's range, NaN, tails and groups without mass; a
    state whose norm is no number."""
    norb, nelec = 10, (5, 4)
    g = inputs.rng(1780)
    v = inputs.random_state(norb, nelec, g)
    flat = v.reshape(-1)
    flat[flat.size // 3:flat.size // 2] = 0
    flat[-300:] = 0
    x = torch.from_numpy(v).cuda().to(dt)
    u = torch.from_numpy(np.concatenate([[0.0, 1.0, -1.0, np.nan, np.nextafter(1.0, 0.0)],
                                         g.random(MANY)])).cuda()
    got = lib.sample_state(x, norb, nelec, uniforms=u)
    assert torch.equal(got[:FEW], lib.sample_state(x, norb, nelec, uniforms=u[:FEW]))
    x.view(-1)[7] = float("inf")
    assert (lib.sample_state(x, norb, nelec, uniforms=u) == -1).all()


@pytest.mark.parametrize("dt,line", [(torch.complex64, 55000 + 69 + 17),
                                     (torch.complex128, 10000 + 241)])
def test_line_between_the_two_forms(lib, dt, line):
    """Calls of one shot either side of the line, by their kernels' count."""
    norb, nelec = 9, (4, 4)  # 63504 / 4 = 15876 amplitudes, 63 groups
    ctx = lib.Context(0)
    v = torch.from_numpy(inputs.random_state(norb, nelec, inputs.rng(1781))).cuda().to(dt)
    u = torch.rand(120000, dtype=torch.float64, device="cuda")
    used = []
    for shots in (line - 200, line + 200):
        ctx.profile_start()
        lib.sample_state(v, norb, nelec, uniforms=u[:shots], ctx=ctx)
        used.append(ctx.profile_stop()["sample_search"][2])
    ctx.close()
    assert used == [1, 6]


def test_scratch_of_many_shots(lib):
    """Ten million shots of a small state: ordered in parts whose scratch stays
    below 80 MB (32 bytes a shot for 2^21 shots at a time, 64 MB, and a few
    2 MB granules of the allocator), the same shots as in one part each."""
    norb, nelec = 10, (5, 5)
    shots = 10_000_000
    g = inputs.rng(1790)
    v = torch.from_numpy(inputs.random_state(norb, nelec, g)).cuda().to(torch.complex64)
    u = torch.rand(shots, dtype=torch.float64, device="cuda")
    ctx = lib.Context(0)
    lib.sample_state(v, norb, nelec, uniforms=u[:1000], ctx=ctx)
    out = torch.empty(shots, dtype=torch.int64, device="cuda")
    del out  # stays in the caching allocator for the call
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    got = lib.sample_state(v, norb, nelec, uniforms=u, ctx=ctx)
    torch.cuda.synchronize()
    assert before - torch.cuda.mem_get_info()[0] < 80 << 20
    for i in (0, 2 ** 21 - 1000, shots - 20000):
        assert torch.equal(got[i:i + 20000], lib.sample_state(v, norb, nelec,
                                                              uniforms=u[i:i + 20000], ctx=ctx))
    ctx.close()


def test_shots_without_room_to_order_them(lib):
    """A call whose scratch cannot be had draws one shot per warp instead."""
    norb, nelec = 10, (5, 5)
    shots = 1_000_000  # 32 MB to order
    g = inputs.rng(1791)
    v = torch.from_numpy(inputs.random_state(norb, nelec, g)).cuda().to(torch.complex64)
    u = torch.rand(shots, dtype=torch.float64, device="cuda")
    ref = lib.sample_state(v, norb, nelec, uniforms=u)
    ctx = lib.Context(0)
    lib.sample_state(v, norb, nelec, uniforms=u[:10], ctx=ctx)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    out = torch.empty(shots, dtype=torch.int64, device="cuda")
    hold = torch.empty(torch.cuda.mem_get_info()[0] - (24 << 20), dtype=torch.uint8, device="cuda")
    try:
        del out
        got = lib.sample_state(v, norb, nelec, uniforms=u, ctx=ctx)
        torch.cuda.synchronize()
    finally:
        del hold
        torch.cuda.empty_cache()
    assert torch.equal(got, ref)
    ctx.close()
