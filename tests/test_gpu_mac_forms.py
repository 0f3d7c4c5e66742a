"""The FP64 translation's forms at the edges of their tiles: leaf boxes that are no
multiple of 16, unions that are no multiple of 8, and 4, 12, 20 and 32
channels (1, 3, 5 and 8 vectors), the tensor-core form against the oracle and against the
register tiles; the mixed form's list translation (one and two units per thread) and
its wide tiles of 8 channels per thread against the register tiles, whose sums they
repeat bit for bit."""
import numpy as np
import pytest

import efie_inputs as E

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def case():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()
    from oracle import fastmv
    from oracle.geometry import build_rwg
    V, T = E.merge_meshes(E.icosphere(8, 0.5, center=(-1.0, 0.0, 0.0)), E.icosphere(6, 0.35, center=(0.9, 0.3, 0.1)))
    k, p, delta, levels = 2 * np.pi, 3, 0.1, 2
    op = fastmv.BsplineEFIE(build_rwg(V, T), k, p, delta, levels)
    X = E.complex_gaussian((8, op.mesh.N), 81)
    return (V, T, k, p, delta, levels), X, {r: op.matvec(X[r]) for r in (0, 4, 7)}


def _products(h, X, variant, n):
    import torch
    h.autotune_set(8, variant, 0)
    return h.matvec(torch.from_numpy(X[:n].copy()).cuda()).cpu().numpy()


def test_fp64_forms(case):
    import paper_2606_13482_gb300 as G
    args, X, ref = case
    _, lv = G.plan(*args)
    assert all(L["n_far_pairs"] > 0 for L in lv) and lv[0]["n_boxes"] % 16
    h = G.EFIE(*args, precision=G.EFIE_FP64)
    try:
        for n in (1, 3, 5, 8):
            a, b = _products(h, X, 0, n), _products(h, X, 1, n)
            # both sum a few hundred terms in 53 bits
            assert np.linalg.norm(a - b) <= 2.0 ** -53 * 100 * np.linalg.norm(b)
            for r in ref:
                if r < n:
                    assert np.linalg.norm(a[r] - ref[r]) < 1e-10 * np.linalg.norm(ref[r])
    finally:
        h.close()


@pytest.mark.parametrize("wide", [False, True])
def test_mixed_lists_repeat_the_tiles(case, wide):
    import paper_2606_13482_gb300 as G
    args, X, _ = case
    if wide:   # more than 64 boxes on the top level
        V, T = E.icosphere(28, 2.0)
        args = (V, T) + args[2:]
        X = E.complex_gaussian((7, 3 * len(T) // 2), 82)
        assert G.plan(*args)[1][-1]["n_boxes"] > 64 and G.plan(*args)[1][0]["n_boxes"] > 64
    h = G.EFIE(*args, precision=G.EFIE_MIXED)
    try:
        for n in (1, 2, 3, 4, 5, 6, 7):
            assert np.array_equal(_products(h, X, 0, n), _products(h, X, 1, n)), n
    finally:
        h.close()


def test_nan_spreads_and_zero_stays(case):
    """A NaN in one vector reaches all of its product, as FP64 arithmetic makes it; a
    zero vector gives zeros."""
    import torch
    import paper_2606_13482_gb300 as G
    args, X, _ = case
    h = G.EFIE(*args, precision=G.EFIE_FP64)
    try:
        x = torch.from_numpy(X.copy()).cuda()
        y0 = h.matvec(x)
        x[3, 7] = float("nan")
        x[5] = 0
        y1 = h.matvec(x)
        assert torch.isnan(torch.view_as_real(y1[3])).any()
        assert not y1[5].abs().any()
        assert torch.equal(y0[[0, 1, 2, 4, 6, 7]], y1[[0, 1, 2, 4, 6, 7]])
    finally:
        h.close()
