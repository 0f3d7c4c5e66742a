"""Device memory of a handle: what the first FP64 product takes."""
import numpy as np
import pytest

import efie_inputs as E

pytestmark = pytest.mark.gpu

K = 2 * np.pi


@pytest.fixture(scope="module")
def G():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()
    import paper_2606_13482_gb300 as G
    return G


def _used():
    import torch
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free, total = torch.cuda.mem_get_info()
    return total - free


def test_fp64_product_takes_its_grids_and_spectra(G):
    """Grids, two spectra and two transform intermediates of 8 vectors, and vectors: the digits
    of the tensor-core translation lie in the intermediates."""
    import torch
    args = (*E.icosphere(28, 1.4), K, 3, 0.1, 2)
    _, lv = G.plan(*args)
    h = G.EFIE(*args, precision=G.EFIE_FP64)
    try:
        x = torch.from_numpy(E.complex_gaussian((8, h.N), 1)).cuda()
        y = torch.empty_like(x)
        before = _used()
        h.matvec(x, y)
        took = _used() - before
        C, Nt = 32, 2 * h.N // 3
        values = sum(2 * L["n_boxes"] * L["sp"] ** 3 * C for L in lv)
        values += 2 * max(L["n_boxes"] * L["nfft"] ** 3 * C for L in lv)
        values += 2 * max(max(L["n_boxes"] * L["nfft"] ** 2 * L["sp"] * C for L in lv),
                          lv[0]["n_boxes"] * lv[1]["sp"] ** 3 * C)   # leaf boxes on the parent's splines
        values += 8 * (3 * h.N + 3 * Nt)
        digits = 24 * 8 * 1.3 * (h.N + Nt)       # of the near field's vectors, columns rounded up to 8
        assert took <= 1.03 * (16 * values + digits), (took, 16 * values, digits)
    finally:
        h.close()


def test_device_bytes_counts_the_digits(G):
    """The digits of a pass of 8 vectors (20 bytes a value and padding) stand in device_bytes in the
    place of the double-float copies (16 bytes a value) that the other near kernels read."""
    import torch
    V, T = E.icosphere(8, 0.5)
    took = []
    for variant in (0, 2):
        h = G.EFIE(V, T, K, 3, 0.1, 2, precision=G.EFIE_MIXED)
        try:
            h.autotune_set(8, 0, variant)
            before = h.info()["device_bytes"]
            h.matvec(torch.from_numpy(E.complex_gaussian((8, h.N), 2)).cuda())
            took.append(h.info()["device_bytes"] - before)
            values = 8 * (h.N + 2 * h.N // 3)
        finally:
            h.close()
    assert 4 * values <= took[0] - took[1] <= 12 * values, (took, values)


def test_refused_solve_leaves_the_products_alone(G):
    """A budget in which a solve's workspace would fit only in part, digits given back or not:
    refused before anything is given back."""
    import torch
    args = (*E.icosphere(8, 0.5), K, 3, 0.1, 2)
    h = G.EFIE(*args, gmres_restart=1)
    x = torch.from_numpy(E.complex_gaussian((16, h.N), 3)).cuda()
    y0 = h.matvec(x)
    resident = h.info()["device_bytes"]
    basis = 16 * 2 * h.N * 16          # 16 right-hand sides, 2 basis vectors; as much again for the rest
    digits = 24 * 8 * (h.N + 2 * h.N // 3)
    h.close()
    h = G.EFIE(*args, gmres_restart=1, device_mem_limit=resident + basis * 3 // 2 - digits * 4 // 3)
    try:
        assert torch.equal(h.matvec(x), y0)
        with pytest.raises(G.EfieError) as e:
            h.solve(x, tol=1e-6)
        assert e.value.code == -2
        assert h.info()["device_bytes"] == resident
        assert torch.equal(h.matvec(x), y0)
    finally:
        h.close()


def test_digits_that_do_not_fit_are_not_tried_again(G):
    """A budget with room for the digits of 8 vectors but not of 64: products of 72, a pass of 64
    and one of 8, keep the smaller digits instead of giving them back and making them again
    (which waits for the device)."""
    import time

    import torch
    args = (*E.icosphere(28, 1.4), K, 3, 0.1, 2)   # two levels that take pairs of 8-vector chunks
    h = G.EFIE(*args, precision=G.EFIE_MIXED)
    h.autotune_set(8, 0, 2)              # double-float copies of the vectors, no digits
    x = torch.from_numpy(E.complex_gaussian((72, h.N), 5)).cuda()
    y = torch.empty_like(x)
    y0 = h.matvec(x)
    # digits of 64 and of 8 vectors take 20 bytes a value, beside the copies' 16 of 64 vectors, and
    # 5 to 20% for columns rounded up to 8
    values = h.N + 2 * h.N // 3
    limit = h.info()["device_bytes"] + 266 * values
    h.close()
    h = G.EFIE(*args, precision=G.EFIE_MIXED, device_mem_limit=limit)
    try:
        for _ in range(2):
            h.matvec(x, y)
        torch.cuda.synchronize()
        assert limit - h.info()["device_bytes"] < 106 * values     # the digits of 8 are there
        t0 = time.perf_counter()
        torch.cuda._sleep(10 ** 9)       # about half a second
        h.matvec(x, y)
        t = time.perf_counter() - t0
        assert t < 0.2, t
        assert float((y - y0).norm() / y0.norm()) < 1e-11
    finally:
        h.close()


@pytest.mark.parametrize("form", ["fp64", "mixed"])
def test_captured_product_keeps_its_buffers(G, form):
    """A caller's CUDA graph of a product, and then a solve that would fit if the digits were given
    back: it is refused, and the replay still computes the product."""
    import torch
    args = (*E.icosphere(8, 0.5), K, 3, 0.1, 2)
    kw = dict(precision=G.EFIE_FP64 if form == "fp64" else G.EFIE_MIXED, gmres_restart=30)
    x = None
    resident = 0
    for limit in (0, 1):
        # room for the basis and two vectors if some 260 kB of the 510 kB and more of digits went
        work = 33 * 16 * 1920 - (1 << 18)
        h = G.EFIE(*args, device_mem_limit=limit and resident + work, **kw)
        try:
            x = torch.from_numpy(E.complex_gaussian((8, h.N), 6)).cuda()
            y = torch.empty_like(x)
            y0 = h.matvec(x)
            resident = h.info()["device_bytes"]
            if not limit:
                continue
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph):
                h.matvec(x, y)
            b = h.rhs_planewave([0, 0, -1.0], [1.0, 0, 0])
            with pytest.raises(G.EfieError) as e:
                h.solve(b, tol=1e-6)
            assert e.value.code == -2 and h.info()["device_bytes"] == resident
            y.zero_()
            graph.replay()
            torch.cuda.synchronize()
            assert torch.equal(y, y0)
            x.mul_(2.0)
            graph.replay()
            torch.cuda.synchronize()
            assert torch.equal(y, 2.0 * y0)
        finally:
            torch.cuda.synchronize()
            h.close()


@pytest.mark.parametrize("form,tol", [("fp64", 1e-13), ("mixed", 1e-11)])
def test_products_without_digits(G, form, tol):
    """A budget just short of the digits: the products run on the other near kernels and agree."""
    import torch
    args = (*E.icosphere(8, 0.5), K, 3, 0.1, 1)
    kw = dict(precision=G.EFIE_FP64 if form == "fp64" else G.EFIE_MIXED)
    h = G.EFIE(*args, **kw)
    x = torch.from_numpy(E.complex_gaussian((8, h.N), 7)).cuda()
    y0 = h.matvec(x)
    values, resident = h.N + 2 * h.N // 3, h.info()["device_bytes"]
    h.close()
    h = G.EFIE(*args, device_mem_limit=resident - 8 * values, **kw)
    try:
        y1 = h.matvec(x)
        # 24 (FP64) or 20 bytes a value and vector less, the 16 of the double-float copies more
        less = 8 * values * (24 if form == "fp64" else 20 - 16)
        assert h.info()["device_bytes"] <= resident - less
        assert not torch.equal(y1, y0) and float((y1 - y0).norm() / y0.norm()) < tol
    finally:
        h.close()


def test_batch_after_a_member_grew(G):
    """A captured batch, then a product of one member that makes its buffers anew: the next batch
    call is recorded again on the new buffers."""
    import torch
    hs = [G.EFIE(*E.icosphere(28, 1.4), K, 3, 0.1, 2, precision=G.EFIE_MIXED),
          G.EFIE(*E.icosphere(6, 0.4), K, 3, 0.1, 1, precision=G.EFIE_MIXED)]
    b = G.Batch(hs)
    try:
        xs = [torch.from_numpy(E.complex_gaussian((1, h.N), 8 + i)).cuda() for i, h in enumerate(hs)]
        ys = [torch.empty_like(x) for x in xs]
        ref = [h.matvec(x) for h, x in zip(hs, xs)]
        for _ in range(2):
            b.matvec(xs, ys)
            torch.cuda.synchronize()
            assert all(torch.equal(y, r) for y, r in zip(ys, ref))
        before = hs[0].info()["device_bytes"]
        hs[0].matvec(torch.from_numpy(E.complex_gaussian((64, hs[0].N), 10)).cuda())
        assert hs[0].info()["device_bytes"] > before
        for y in ys:
            y.zero_()
        b.matvec(xs, ys)
        torch.cuda.synchronize()
        assert all(torch.equal(y, r) for y, r in zip(ys, ref))
    finally:
        torch.cuda.synchronize()
        b.close()
        for h in hs:
            h.close()
