"""Transfers by the nonzeros of their matrices against the oracle where the rule's
two sides meet: degrees 3 (fused in both precisions), 4 and 6 (fused in FP64 and,
downward, in FP32) on a two-level tree with far pairs on both levels, some parents
with few children, for 1, 3 and 8 right-hand sides (the smallest and largest
channel counts)."""
import numpy as np
import pytest

import efie_inputs as E

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p", [3, 4, 6])
def test_fused_transfers(p):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()
    import paper_2606_13482_gb300 as G
    from oracle import fastmv
    from oracle.geometry import build_rwg
    V, T = E.merge_meshes(E.icosphere(7, 0.45, center=(-0.9, 0.0, 0.0)), E.icosphere(6, 0.4, center=(0.9, 0.3, 0.1)))
    k, delta, levels = 2 * np.pi, 0.1, 2
    _, lv = G.plan(V, T, k, p, delta, levels)
    assert len(lv) == 2 and all(L["n_far_pairs"] > 0 for L in lv)
    op = fastmv.BsplineEFIE(build_rwg(V, T), k, p, delta, levels)
    X = E.complex_gaussian((8, op.mesh.N), 60 + p)
    ref = {r: op.matvec(X[r]) for r in (0, 2, 7)}
    for form, tol in ((G.EFIE_FP64, 1e-10), (G.EFIE_MIXED, 1e-5)):   # the forms' gates against the oracle
        h = G.EFIE(V, T, k, p, delta, levels, precision=form)
        try:
            for n in (1, 3, 8):
                Y = h.matvec(torch.from_numpy(X[:n].copy()).cuda()).cpu().numpy()
                for r in ref:
                    if r < n:
                        assert np.linalg.norm(Y[r] - ref[r]) / np.linalg.norm(ref[r]) < tol, (p, form, n, r)
        finally:
            h.close()
