"""Plane-wave right-hand sides at the edges of their forms: one wave and the most
that take the direct sums, the fewest by leaf box, a count that is no multiple of the
waves per block, elements small enough for the power series and too large for them
(lambda / 3), and a box of 2,880 triangles, against the oracle's rule; that up to 64
waves have the bits of the direct sums, which do not depend on the boxes; and that
more have them where a box's triangles do not fit in shared memory."""
import numpy as np
import pytest

import efie_inputs as E

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("freq,radius,delta,n", [(5, 0.3, 0.1, 1), (5, 0.3, 0.1, 65), (5, 0.3, 0.1, 83),
                                                 (3, 0.9, 0.45, 70), (12, 0.04, 0.3, 3)])
def test_planewave_boxes(freq, radius, delta, n):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()
    import paper_2606_13482_gb300 as G
    from oracle.dense import rhs_planewave
    from oracle.geometry import build_rwg
    V, T = E.icosphere(freq, radius, center=(0.3, -0.2, 0.1))
    k = 2 * np.pi
    rng = np.random.default_rng(freq)
    khat = rng.standard_normal((n, 3))
    khat /= np.linalg.norm(khat, axis=1, keepdims=True)
    pol = np.cross(khat, rng.standard_normal((n, 3)))
    h = G.EFIE(V, T, k, 3, delta, 1)
    try:
        got = h.rhs_planewave(khat, pol).cpu().numpy()
    finally:
        h.close()
    ref = rhs_planewave(build_rwg(V, T), k, khat, pol)
    # 36 rounded terms of size |p| h and phases of a few radians: a few 1e-15 of the norm
    err = np.linalg.norm(got - ref, axis=1) / np.linalg.norm(ref, axis=1)
    print(f"plane waves, freq {freq}, radius {radius}: {err.max():.2e}")
    assert err.max() < 3e-14


@pytest.mark.parametrize("freq,radius,n,deltas", [(5, 0.3, 1, (0.1, 0.15)), (5, 0.3, 64, (0.1, 0.15)),
                                                  (12, 0.04, 66, (0.3,))])
def test_direct_bits(freq, radius, n, deltas):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()
    import paper_2606_13482_gb300 as G
    V, T = E.icosphere(freq, radius)
    rng = np.random.default_rng(n)
    khat = rng.standard_normal((n, 3))
    khat /= np.linalg.norm(khat, axis=1, keepdims=True)
    pol = np.cross(khat, rng.standard_normal((n, 3)))
    got = []
    for delta in deltas:
        h = G.EFIE(V, T, 2 * np.pi, 3, delta, 1)
        got.append(h.rhs_planewave(khat, pol).cpu().numpy())
        got.append(np.concatenate([h.rhs_planewave(khat[i:i + 2], pol[i:i + 2]).cpu().numpy() for i in range(0, n, 2)]))
        h.close()
    assert all((y == got[0]).all() for y in got)
