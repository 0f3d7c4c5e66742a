"""Digit products (near field, FP64 translation) of vectors near the ends of the FP64
range: scaling a vector by a power of two scales its product, down to results that are
subnormal numbers."""
import numpy as np
import pytest

import efie_inputs as E

pytestmark = pytest.mark.gpu

K = 2 * np.pi
# rounding of a few hundred terms whose two parts nearly cancel, 53 bits; the digits
# themselves do not depend on the power of two
TOL = 2.0 ** -53 * 1e3


def _case(name):
    if name == "near":   # all boxes adjacent
        return (*E.icosphere(5, 0.3), K, 3, 0.15, 1)
    return (*E.merge_meshes(E.icosphere(8, 0.5, center=(-1.0, 0.0, 0.0)), E.icosphere(6, 0.35, center=(0.9, 0.3, 0.1))),
            K, 3, 0.1, 2)


def _scaled(x, e):
    return x * 2.0 ** (e // 2) * 2.0 ** (e - e // 2)


@pytest.mark.parametrize("name,form", [("near", "fp64"), ("near", "mixed"), ("far", "fp64")])
def test_powers_of_two(name, form):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()
    import paper_2606_13482_gb300 as G
    h = G.EFIE(*_case(name), precision=G.EFIE_FP64 if form == "fp64" else G.EFIE_MIXED)
    try:
        X = E.complex_gaussian((8, h.N), 7)
        X[1] *= 2.0 ** -np.linspace(0, 40, h.N)
        X[2] = 0
        X = torch.from_numpy(X).cuda()
        Y = h.matvec(X).cpu().numpy()
        for e in (-960, -980, -1000, 900):
            Z = _scaled(h.matvec(_scaled(X, e)).cpu().numpy(), -e)
            for r in range(8):
                assert np.linalg.norm(Z[r] - Y[r]) <= TOL * np.linalg.norm(Y[r]), (e, r)
        # subnormal inputs and results: within a few hundred roundings to 2^-1074, times
        # the factors k and 1 / k of the two parts
        x = _scaled(X, -1030)
        y = _scaled(h.matvec(_scaled(x, 1030)).cpu().numpy(), -1030)
        z = h.matvec(x).cpu().numpy()
        assert np.abs(y).max() > 2.0 ** -1040 and np.abs(z - y).max() <= 2000 * 2.0 ** -1074
    finally:
        h.close()


@pytest.mark.parametrize("form,tol", [("fp64", TOL), ("mixed", 2.0 ** -48 * 1e3)])
def test_graded_vectors(form, tol):
    """Entries of one box from 1 to 2^-60: the digits hold 60 (FP64) or 50 bits below a box's
    largest entry, so the product keeps the bound of ungraded vectors."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()
    import paper_2606_13482_gb300 as G
    from oracle import dense
    from oracle.geometry import build_rwg
    args = _case("near")
    ref = dense.efie_matrix(build_rwg(*args[:2]), K)
    h = G.EFIE(*args, precision=G.EFIE_FP64 if form == "fp64" else G.EFIE_MIXED)
    try:
        X = E.complex_gaussian((4, h.N), 9)
        rng = np.random.default_rng(11)
        for r, bits in enumerate((20, 40, 60)):
            X[r] *= 2.0 ** -rng.uniform(0, bits, h.N)
        X[3] *= 1e-12
        X[3, h.N // 3] = 1.0
        Y = h.matvec(torch.from_numpy(X).cuda()).cpu().numpy()
        for r in range(4):
            y = ref @ X[r]
            err = np.linalg.norm(Y[r] - y) / np.linalg.norm(y)
            print(f"graded vector {r}, {form}: {err:.2e}")
            assert err <= tol
    finally:
        h.close()
