"""Mode products along long axes (the tiled kernels): a two-level tree with 23
leaf splines per axis, so that the transforms take 27 and 47 splines, the upward
transfer 27 -> 47 and the downward one 47 -> 27, for 1, 3 and 8 right-hand sides
(4, 12 and 32 channels), against the oracle; and the anterpolation's lane forms
(1, 2, 4 and 8 lanes a point) on the same boxes."""
import numpy as np
import pytest

import efie_inputs as E

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-10, "mixed": 1e-5}   # the forms' gates against the oracle


@pytest.fixture(scope="module")
def case():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()
    from oracle import fastmv
    from oracle.geometry import build_rwg
    V, T = E.merge_meshes(E.icosphere(5, 0.4, center=(-1.7, 0.0, 0.0)), E.icosphere(5, 0.4, center=(1.7, 0.3, 0.1)))
    X = E.complex_gaussian((8, 3 * len(T) // 2), 77)
    op = fastmv.BsplineEFIE(build_rwg(V, T), 2 * np.pi, 3, 0.045, 2, n_splines=23)
    return V, T, X, {r: op.matvec(X[r]) for r in (0, 1, 2, 7)}


@pytest.mark.parametrize("form", ["fp64", "mixed"])
def test_long_axes(case, form):
    import torch
    import paper_2606_13482_gb300 as G
    V, T, X, ref = case
    o = G.Options()
    o.n_splines = 23
    _, lv = G.plan(V, T, 2 * np.pi, 3, 0.045, 2, o)
    assert [L["sp"] for L in lv] == [27, 47] and all(L["n_far_pairs"] > 0 for L in lv)
    h = G.EFIE(V, T, 2 * np.pi, 3, 0.045, 2, n_splines=23,
               precision=G.EFIE_FP64 if form == "fp64" else G.EFIE_MIXED)
    try:
        for n in (1, 2, 3, 8):
            Y = h.matvec(torch.from_numpy(X[:n].copy()).cuda()).cpu().numpy()
            for r in ref:
                if r < n:
                    err = np.linalg.norm(Y[r] - ref[r]) / np.linalg.norm(ref[r])
                    print(f"long axes, {form}, {n} vectors, {r}: {err:.2e}")
                    assert err < TOL[form]
    finally:
        h.close()


def test_anterpolation_forms():
    """The FP64 lane forms on boxes whose functions are staged whole (1 to 4 vectors)
    and in several passes over the sorted lists (8 vectors): 735 RWGs a box."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()
    import paper_2606_13482_gb300 as G
    V, T = E.merge_meshes(E.icosphere(14, 0.4, center=(-1.7, 0.0, 0.0)), E.icosphere(14, 0.4, center=(1.7, 0.3, 0.1)))
    args = (V, T, 2 * np.pi, 3, 0.2, 1)
    assert G.plan(*args)[1][0]["n_far_pairs"] > 0
    X = torch.from_numpy(E.complex_gaussian((8, 3 * len(T) // 2), 5)).cuda()
    h = G.EFIE(*args, precision=G.EFIE_FP64)
    try:
        one = torch.cat([h.matvec(X[r:r + 1].contiguous()) for r in range(8)])
        for n in (2, 3, 4, 5, 8):
            y = h.matvec(X[:n].contiguous())
            # both sum lists of up to some hundred rounded terms in 53 bits
            assert (y - one[:n]).norm() <= 2.0 ** -53 * 100 * one[:n].norm(), n
    finally:
        h.close()
