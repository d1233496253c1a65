"""Contexts of several threads, each on its own stream and sector: the same
results as alone, and no launch fails for what another thread does."""

import os
import threading

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


def _work(lib, kind, norb, nelec, dt, n):
    ctx = lib.Context(0)
    ctx.set_rotation_path(lib.FS_ROT_GIVENS)
    g = inputs.rng(44000 + norb)
    U = inputs.haar_unitary(norb, g)
    h1, h2 = g.normal(0, 1, (norb, norb)), g.normal(0, 1, (norb,) * 4)
    v = torch.from_numpy(inputs.random_state(norb, nelec, g)).cuda().to(dt)
    with torch.cuda.stream(torch.cuda.Stream()):
        for _ in range(n):
            if kind == "operator":
                out = lib.apply_molecular_hamiltonian(v, h1, h2, norb, nelec, ctx=ctx)
            else:
                out = lib.apply_orbital_rotation(v, U, norb, nelec, ctx=ctx)
        torch.cuda.current_stream().synchronize()
    ctx.close()
    return out.cpu().numpy()


@pytest.mark.parametrize("kind,dt,sectors", [
    ("operator", torch.complex64, [(6, (3, 3)), (10, (5, 5)), (10, (2, 2)), (9, (4, 4))]),
    ("operator", torch.complex128, [(6, (3, 3)), (10, (5, 5)), (10, (2, 2)), (9, (4, 4))]),
    ("rotation", torch.complex64, [(9, (4, 5)), (11, (5, 5)), (12, (6, 2)), (10, (5, 3))]),
    ("rotation", torch.complex128, [(9, (4, 5)), (11, (5, 5)), (12, (6, 2)), (10, (5, 3))])])
def test_contexts_of_several_threads(lib, kind, dt, sectors):
    alone = [_work(lib, kind, n, e, dt, 1) for n, e in sectors]
    out, errors = [None] * len(sectors), []

    def run(i):
        try:
            out[i] = _work(lib, kind, *sectors[i], dt, 400)
        except Exception as e:  # noqa: BLE001 - reported by the test's own thread
            errors.append(e)
    threads = [threading.Thread(target=run, args=(i,)) for i in range(len(sectors))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for a, b in zip(alone, out):
        assert np.array_equal(a, b)
