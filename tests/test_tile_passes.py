"""GPU: the tile kernels of spatially ordered lists against the passes they take the place of."""
import numpy as np
import pytest

from paper_2011_14984_gb300 import ics

pytestmark = pytest.mark.gpu


def _frost(*args, **kw):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2011_14984_gb300.frost import Frost
    return Frost(*args, **kw)


@pytest.mark.parametrize("sym", [0, 1, 2])
@pytest.mark.parametrize("n,masses", [(16384, "equal"), (16417, "kroupa"), (20001, "binaries"), (16385, "rest")])
def test_tiled_timesteps_are_those_of_every_pair(n, masses, sym):
    # the minimum over the same FP32 pair values as the one-sided and the symmetric pass, which
    # sets below the tile kernels' size take: every pair of particles is in the union of two of
    # five chunks, and the least of its unions' steps is a particle's step over all, bit for bit
    import torch
    if masses == "binaries":
        m, x, v = ics.plummer_kroupa_binaries(n, 11)
    else:
        m, x, v = ics.plummer(n, 11, ics.kroupa_masses(n, 11) if masses == "kroupa" else None)
    if masses == "rest":
        # pairs almost at rest relative to each other, far apart: their symmetrised fly-by steps
        # are the smallest of all, and no box shows them
        v[: n // 2] = 0.0
        v[: n // 2, 0] = 1e-9 * np.arange(n // 2)
    f = _frost(m, x, v, sym=sym)
    tau = f.timesteps().cpu().numpy()
    perm = np.random.default_rng(3).permutation(n).astype(np.int32)
    tau_p = f.timesteps(torch.from_numpy(perm).cuda()).cpu().numpy()
    assert np.array_equal(tau_p, tau[perm])
    ref = np.full(n, np.inf)
    chunks = np.array_split(np.arange(n, dtype=np.int32), 5)
    for a in range(5):
        for b in range(a):
            u = np.concatenate([chunks[b], chunks[a]])
            ref[u] = np.minimum(ref[u], f.timesteps(torch.from_numpy(u).cuda()).cpu().numpy())
    assert np.array_equal(tau, ref)


def test_step_from_an_ordered_set_is_deterministic_and_restartable():
    n = 16384
    m, x, v = ics.plummer(n, 4)
    f = _frost(m, x, v)
    f.step(2.0 ** -9, 2)
    xa, va, _ = f.state()
    g = _frost(m, x, v)
    g.step(2.0 ** -9, 1)
    xm, vm, t = g.state()
    h = _frost(m, xm, vm)
    h.set_state(t=t)
    h.step(2.0 ** -9, 1)
    xb, vb, _ = h.state()
    assert np.array_equal(xa, xb) and np.array_equal(va, vb)
