"""Near-field assembly with the phases of a triangle pair as power series: element
sizes in each of its ranges (eight terms, ten terms, full sine and cosine), FP64
form on one-level trees whose boxes are all adjacent, against the dense EFIE."""
import numpy as np
import pytest

import efie_inputs as E

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("freq,radius", [(4, 0.15), (3, 0.3), (2, 0.9)])   # longest edges about 0.045, 0.12, 0.55
def test_assembly_series(freq, radius):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()
    import paper_2606_13482_gb300 as G
    from oracle import dense
    from oracle.geometry import build_rwg
    V, T = E.icosphere(freq, radius)
    k = 2 * np.pi
    m = build_rwg(V, T)
    A, Vm = dense.assemble_dense(m, k)
    X = E.complex_gaussian((2, m.N), freq)
    h = G.EFIE(V, T, k, 3, 0.5 * radius, 1)
    try:
        yA, yV = (t.cpu().numpy() for t in h.matvec_parts(torch.from_numpy(X).cuda()))
    finally:
        h.close()
    rho = m.sigmaT_apply(X)
    for r in range(2):
        a, v = A @ X[r], m.sigma_apply(Vm @ rho[r])
        ea, ev = np.linalg.norm(yA[r] - a) / np.linalg.norm(a), np.linalg.norm(yV[r] - v) / np.linalg.norm(v)
        print(f"assembly, freq {freq}, radius {radius}: A {ea:.2e}, V {ev:.2e}")
        # entries of a few 1e-16 of their size, sums of a few hundred of them that nearly cancel (by up to 100)
        assert ea < 2.0 ** -53 * 1e3 and ev < 2.0 ** -53 * 1e3
