"""The FP32 transform passes at the edges of their forms: spline counts of every
degree (lines of 9, 13 and 21 outputs, and shorter ones), 1, 3 and 8 right-hand
sides (4, 12 and 32 channels) and the line and the fused schedules, against the
FP64 handle's product."""
import numpy as np
import pytest

import efie_inputs as E

pytestmark = pytest.mark.gpu

TOL = 1e-5   # the mixed form's gate against FP64


@pytest.mark.parametrize("p", [1, 2, 3, 4, 6])
def test_transform_forms(p):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()
    import paper_2606_13482_gb300 as G
    V, T = E.merge_meshes(E.icosphere(7, 0.45, center=(-0.9, 0.0, 0.0)), E.icosphere(6, 0.4, center=(0.9, 0.3, 0.1)))
    args = (V, T, 2 * np.pi, p, 0.1, 2)
    assert all(L["n_far_pairs"] > 0 for L in G.plan(*args)[1])
    x = torch.from_numpy(E.complex_gaussian((8, 3 * len(T) // 2), p)).cuda()
    h = G.EFIE(*args, precision=G.EFIE_FP64)
    ref = h.matvec(x).cpu().numpy()
    h.close()
    h = G.EFIE(*args, precision=G.EFIE_MIXED)
    try:
        for schedule in (0, 2, 3):
            h.transform_schedule(schedule)
            for n in (1, 3, 8):
                y = h.matvec(x[:n].contiguous()).cpu().numpy()
                err = np.linalg.norm(y - ref[:n], axis=1) / np.linalg.norm(ref[:n], axis=1)
                print(f"p = {p}, schedule {schedule}, {n} vectors: {err.max():.2e}")
                assert err.max() < TOL
    finally:
        h.close()
