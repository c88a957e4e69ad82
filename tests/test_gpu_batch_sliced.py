"""Batches through sliced launches (slice.cu) against the oracle: levels below
and above the launches' tile depth, single and several launches per fractal,
uneven generation counts, two rules, unaligned buffers, instances next to each
other in memory, and instances that the tile kernels keep."""
import numpy as np
import pytest
import torch

import oracle
from paper_2110_12952_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("seed,even", [(1, True), (2, False), (3, False)])
def test_uneven_sliced_batches(seed, even):
    from paper_2110_12952_gb300 import Batch, Fractal
    rng = np.random.default_rng(seed)
    levels = {"triangle": (1, 12), "carpet": (1, 6), "vicsek": (2, 8), "h_fractal": (3, 5), "menger": (3, 3)}
    specs = []
    for i in range(70):
        name = list(levels)[int(rng.integers(0, len(levels)))]
        lo, hi = levels[name]
        steps = 7 if even else int(rng.integers(0, 25))
        rule = W.default_rule(W.FAMILIES[name]) if i % 5 else (W.rule_masks([2], [1, 2, 3]) if name != "menger" else W.MENGER_B5S45)
        specs.append((W.FAMILIES[name], int(rng.integers(lo, hi + 1)), steps, rule, int(rng.integers(0, 3))))
    handles, batch, bufs = {}, Batch(), []
    total = sum(f.k ** r + 40 for f, r, _, _, _ in specs)
    src = torch.zeros(total, dtype=torch.uint8, device="cuda")
    dst = torch.full((total,), 77, dtype=torch.uint8, device="cuda")
    pos = 0
    for i, (fam, r, steps, rule, skew) in enumerate(specs):
        if (fam.name, r) not in handles:
            handles[fam.name, r] = (Fractal.from_family(fam, r), oracle.Fractal(fam.k, fam.s, r, fam.dim, fam.table()))
        g, o = handles[fam.name, r]
        pos = (pos + 15) // 16 * 16 + skew
        x, y = src[pos:pos + g.cells], dst[pos:pos + g.cells]
        x.copy_(torch.from_numpy(o.init_bernoulli(i, 0.45)))
        batch.add(g, x, y, steps, rule=rule)
        bufs.append((pos, g.cells))
        pos += g.cells
    for rep in range(2):
        batch.run()
        torch.cuda.synchronize()
        got = dst.cpu().numpy().copy()
        for i, ((fam, r, steps, rule, _), (p, n)) in enumerate(zip(specs, bufs)):
            o = handles[fam.name, r][1]
            want = o.step(o.init_bernoulli(i + 1000 * rep, 0.45), rule=oracle.Rule(*rule), steps=steps)
            assert np.array_equal(got[p:p + n], want), (fam.name, r, steps, i)
            got[p:p + n] = 77
        assert (got == 77).all()    # nothing written between the instances
        for i, ((fam, r, _, _, _), (p, n)) in enumerate(zip(specs, bufs)):
            src[p:p + n].copy_(torch.from_numpy(handles[fam.name, r][1].init_bernoulli(i + 1000, 0.45)))
    batch.close()
    for g, _ in handles.values():
        g.check()
        g.close()


@pytest.mark.parametrize("name,r", [("triangle", 8), ("carpet", 5), ("h_fractal", 4)])
def test_a_batch_readies_its_handles(name, r):
    # what a batch run has always made possible: the allocation-free step and a captured generation of a handle whose
    # only call so far was the batch
    from paper_2110_12952_gb300 import Batch, Fractal
    fam = W.FAMILIES[name]
    g, o = Fractal.from_family(fam, r), oracle.Fractal(fam.k, fam.s, r, fam.dim, fam.table())
    v = o.init_bernoulli(4, 0.45)
    x = torch.from_numpy(v).cuda()
    y, z, t = torch.empty_like(x), torch.empty_like(x), torch.empty_like(x)
    batch = Batch()
    batch.add(g, x, y, 4)
    batch.run()
    birth, survive = W.LIFE_B3S23
    assert g._lib.fractal_step_noalloc(g._h, x.data_ptr(), z.data_ptr(), 3, birth, survive, 0) == 0
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        g.step(x, out=t, steps=1)
    graph.replay()
    torch.cuda.synchronize()
    for got, n in ((y, 4), (z, 3), (t, 1)):
        assert np.array_equal(got.cpu().numpy(), o.step(v, steps=n)), n
    del graph
    batch.close()
    g.check()
    g.close()


def test_copies_come_before_generations():
    # an instance of no generations normalises its input into another instance's input; one of a single generation
    # reads what an instance of four overwrites from its second generation on
    from paper_2110_12952_gb300 import Batch, Fractal
    fam = W.TRIANGLE
    g, o = Fractal.from_family(fam, 9), oracle.Fractal(fam.k, fam.s, 9, fam.dim, fam.table())
    v, w = o.init_bernoulli(1, 0.45), o.init_bernoulli(2, 0.45)
    p, q = torch.from_numpy(v * 7).cuda(), torch.from_numpy(w).cuda()
    x, y, z = torch.zeros_like(p), torch.zeros_like(p), torch.zeros_like(p)
    batch = Batch()
    batch.add(g, x, y, 3)     # reads the copy
    batch.add(g, p, x, 0)     # the copy
    batch.add(g, q, z, 1)     # reads q before ...
    batch.add(g, p, q, 4)     # ... this instance writes it
    batch.run()
    torch.cuda.synchronize()
    assert np.array_equal(x.cpu().numpy(), v)
    assert np.array_equal(y.cpu().numpy(), o.step(v, steps=3))
    assert np.array_equal(z.cpu().numpy(), o.step(w, steps=1))
    assert np.array_equal(q.cpu().numpy(), o.step(v, steps=4))
    batch.close()
    g.close()
