"""The tensor-core near field (digits of 10 bits, FP16 MMAs) at the edges of its
tiles: counts of right-hand sides around its 8-, 16-, 32- and 64-vector forms,
rows and columns that are no multiples of 16 and 8, vectors far from 1 in
magnitude, zero vectors, and a NaN in one vector.  One-level trees whose boxes
are all adjacent, so that the product is the near field alone, against the
dense EFIE."""
import numpy as np
import pytest

import efie_inputs as E

pytestmark = pytest.mark.gpu

K = 2 * np.pi
# A row's entries and x carry 48 bits (mixed) or 53 (FP64) below their largest
# values; the two parts of T nearly cancel on these small spheres (by about
# 100), and a sum of a few hundred rounded terms grows by about 10.
TOL = {"mixed": 2.0 ** -48 * 1e3, "fp64": 2.0 ** -53 * 1e3}


@pytest.fixture(scope="module")
def G():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()
    import paper_2606_13482_gb300 as G
    return G


@pytest.fixture(scope="module", params=[(3, 0.15), (5, 0.3)])   # 270 and 750 RWG: 34 and 94 a box on average
def problem(request):
    from oracle import dense
    from oracle.geometry import build_rwg
    freq, radius = request.param
    V, T = E.icosphere(freq, radius)
    return V, T, dense.efie_matrix(build_rwg(V, T), K), 0.5 * radius


@pytest.mark.parametrize("form", ["mixed", "fp64"])
def test_counts_and_scales(G, problem, form):
    import torch
    V, T, ref, delta = problem
    h = G.EFIE(V, T, K, 3, delta, 1, precision=G.EFIE_FP64 if form == "fp64" else G.EFIE_MIXED)
    try:
        for n in (1, 2, 7, 8, 9, 16, 17, 32, 33, 64, 65):
            X = E.complex_gaussian((n, h.N), 10 + n)
            X *= 2.0 ** np.linspace(-60, 60, n)[:, None]
            if n > 2:
                X[1] = 0.0
            Y = h.matvec(torch.from_numpy(X).cuda()).cpu().numpy()
            for r in range(n):
                y = ref @ X[r]
                scale = np.linalg.norm(y)
                err = np.linalg.norm(Y[r] - y)
                assert err <= TOL[form] * scale, (n, r, err / max(scale, 1e-300))
    finally:
        h.close()


@pytest.mark.parametrize("form", ["mixed", "fp64"])
def test_nan_stays_in_its_vector(G, problem, form):
    import torch
    V, T, _, delta = problem
    h = G.EFIE(V, T, K, 3, delta, 1, precision=G.EFIE_FP64 if form == "fp64" else G.EFIE_MIXED)
    try:
        X = torch.from_numpy(E.complex_gaussian((9, h.N), 3)).cuda()
        y0 = h.matvec(X)
        X[4, 5] = float("nan")
        y1 = h.matvec(X)
        assert torch.isnan(torch.view_as_real(y1[4])).any()
        keep = [r for r in range(9) if r != 4]
        assert torch.equal(y0[keep], y1[keep])
    finally:
        h.close()


def test_digit_buffers_are_given_back(G):
    """A memory limit that leaves no room for the digits of x: the products run
    on the other near kernels and agree."""
    import torch
    V, T = E.icosphere(8, 0.5)
    h = G.EFIE(V, T, K, 3, 0.1, 1, precision=G.EFIE_MIXED)
    x = torch.from_numpy(E.complex_gaussian((3, h.N), 4)).cuda()
    y0 = h.matvec(x)
    # what products need, and double-float copies of 8 work vectors; the digits of
    # x take half as much again
    limit = h.info()["device_bytes"] + (h.N + 2 * h.N // 3) * 8 * 16 + (1 << 14)
    h.close()
    h = G.EFIE(V, T, K, 3, 0.1, 1, precision=G.EFIE_MIXED, device_mem_limit=limit)
    try:
        y1 = h.matvec(x)
        assert float((y1 - y0).norm() / y0.norm()) < 1e-11
    finally:
        h.close()
