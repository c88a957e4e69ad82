"""The maps and the box views through tables (maps.cu) against the oracle:
arrays long enough for the tables, levels that do and do not divide into whole
groups, fractals whose first digit tuple is and is not a replica, indices
beyond 2^31, points off the fractal and outside the box, odd counts, and
buffers that are only aligned to their type."""
import numpy as np
import pytest
import torch

import oracle
from paper_2110_12952_gb300 import workloads as W

pytestmark = pytest.mark.gpu

N = 1000001   # from 2e7 points x levels x replicas on the maps use tables
CASES = [("triangle", 1), ("triangle", 7), ("triangle", 13), ("triangle", 20), ("carpet", 3), ("carpet", 9), ("vicsek", 4),
         ("vicsek", 12), ("menger", 2), ("menger", 5), ("menger", 7), ("candy", 7), ("x_fractal", 11), ("full_square", 15),
         ("cantor_set", 19)]


@pytest.mark.parametrize("name,r", CASES)
@pytest.mark.parametrize("skew", [0, 1])
def test_long_map_arrays(name, r, skew):
    from paper_2110_12952_gb300 import Fractal
    fam = W.FAMILIES[name]
    g, o = Fractal.from_family(fam, r), oracle.Fractal(fam.k, fam.s, r, fam.dim, fam.table())
    rng = np.random.default_rng(r)
    w = rng.integers(0, o.cells, N, dtype=np.int64)
    w[:4] = (0, o.cells - 1, -1, o.cells)
    buf = torch.empty(N + skew, dtype=torch.int64, device="cuda")[skew:]
    buf.copy_(torch.from_numpy(w))
    out = torch.empty((N + skew) * fam.dim, dtype=torch.int32, device="cuda")[skew * fam.dim:].view(N, fam.dim)
    lam = g.lam(buf, out=out).cpu().numpy()
    want = np.full((N, fam.dim), -1, dtype=np.int64)
    ok = (w >= 0) & (w < o.cells)
    want[ok] = o.lam(w[ok])
    assert np.array_equal(lam, want)
    # the points' neighbours, random points and points outside
    c = lam.copy()
    c[ok] += rng.integers(-1, 2, (int(ok.sum()), fam.dim), dtype=np.int32)
    c[5:9] = (-1, 0, o.side, 2**31 - 1)[:1]
    c[9:200] = rng.integers(0, o.side, (191, fam.dim))
    c[200:204, 0] = (-(2**31), -5, o.side - 1, o.side)
    cb = torch.empty((N + skew) * fam.dim, dtype=torch.int32, device="cuda")[skew * fam.dim:].view(N, fam.dim)
    cb.copy_(torch.from_numpy(c))
    nu = torch.empty(N + skew, dtype=torch.int64, device="cuda")[skew:]
    n2 = torch.empty((N + skew) * fam.dim, dtype=torch.int64, device="cuda")[skew * fam.dim:].view(N, fam.dim)
    assert np.array_equal(g.nu(cb, out=nu).cpu().numpy(), o.nu(c))
    assert np.array_equal(g.nu2d(cb, out=n2).cpu().numpy(), o.nu2d(c))
    # the same points many times over: the tables grow with the array
    many = 13
    for fn, x, y in ((g.lam, buf, out), (g.nu, cb, nu), (g.nu2d, cb, n2)):
        big = fn(x.repeat(*((many,) + (1,) * (x.dim() - 1))))
        assert bool((big.view(many, *y.shape) == y).all())
    g.close()


@pytest.mark.parametrize("name,r", [("triangle", 11), ("triangle", 12), ("carpet", 6), ("vicsek", 7), ("menger", 4), ("candy", 5),
                                    ("full_square", 8)])
def test_box_views_by_tiles(name, r):
    from paper_2110_12952_gb300 import Fractal
    fam = W.FAMILIES[name]
    g, o = Fractal.from_family(fam, r), oracle.Fractal(fam.k, fam.s, r, fam.dim, fam.table())
    x = o.init_bernoulli(3, 0.5)
    x[::5] *= 9
    idx = o.lam(np.arange(o.cells)) @ (o.side ** np.arange(fam.dim))
    for off in (0, 3):
        src = torch.empty(o.cells + off, dtype=torch.uint8, device="cuda")[off:]
        src.copy_(torch.from_numpy(x))
        box = torch.full((o.box_cells + off,), 5, dtype=torch.uint8, device="cuda")[off:]
        g.scatter(src, out=box)
        want = np.zeros(o.box_cells, dtype=np.uint8)
        want[idx] = x != 0
        assert np.array_equal(box.cpu().numpy(), want)
        box += 2 * box   # members alive: 3
        back = torch.full((o.cells + off,), 5, dtype=torch.uint8, device="cuda")[off:]
        assert np.array_equal(g.gather(box, out=back).cpu().numpy(), (x != 0).astype(np.uint8))
    g.close()


@pytest.mark.parametrize("name,r", [("carpet", 9), ("full_square", 14), ("menger", 5)])
def test_large_boxes_filled(name, r):
    # rows shorter and longer than a block's run of 16384 cells: every cell is where gather finds it, nothing elsewhere
    from paper_2110_12952_gb300 import Fractal
    g = Fractal.from_family(W.FAMILIES[name], r)
    x = torch.empty(g.cells, dtype=torch.uint8, device="cuda").bernoulli_(0.5)
    box = torch.full((g.box_cells,), 9, dtype=torch.uint8, device="cuda")
    g.scatter(x, out=box)
    assert torch.equal(g.gather(box), x)
    assert int(box.max()) == 1 and int(box.sum(dtype=torch.int64)) == int(x.sum(dtype=torch.int64))
    g.close()


@pytest.mark.parametrize("name,r", [("triangle", 12), ("carpet", 7), ("h_fractal", 7), ("full_square", 10), ("menger", 5), ("candy", 6)])
def test_longer_box_views_by_tiles(name, r):
    # states from the length on at which the views go by tiles, against the oracle, at any address
    test_box_views_by_tiles(name, r)


@pytest.mark.parametrize("name,r", [("triangle", 20), ("carpet", 9), ("menger", 6), ("vicsek", 12)])
def test_largest_coordinates_are_outside(name, r):
    # coordinates up to the type's ends, along each axis, in arrays that go through tables
    from paper_2110_12952_gb300 import Fractal
    fam = W.FAMILIES[name]
    g, o = Fractal.from_family(fam, r), oracle.Fractal(fam.k, fam.s, r, fam.dim, fam.table())
    rng = np.random.default_rng(r)
    c = o.lam(rng.integers(0, o.cells, N, dtype=np.int64)).astype(np.int32)
    ends = np.array([2**31 - 1, 2**31 - 2, -2**31, -1, o.side, o.side - 1, 0, 1 << 30, -(1 << 30)], dtype=np.int32)
    for a in range(fam.dim):
        c[a * 5000:(a + 1) * 5000 - 1000, a] = np.resize(ends, 4000)
    c[20000:24000] = ends[rng.integers(0, len(ends), (4000, fam.dim))]
    d = torch.from_numpy(c).cuda()
    assert np.array_equal(g.nu(d).cpu().numpy(), o.nu(c))
    assert np.array_equal(g.nu2d(d).cpu().numpy(), o.nu2d(c))
    g.close()
