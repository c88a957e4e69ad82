"""Box generations through packed words (bb.cu) against the oracle: sides that
are and are not whole words, rows that start at any byte, one and several
words per row, bytes other than 0 and 1 on and off the fractal, the two rules
with a closed form and others, one and several generations."""
import numpy as np
import pytest
import torch

import oracle
from paper_2110_12952_gb300 import workloads as W

pytestmark = pytest.mark.gpu

CASES = [("triangle", 5), ("triangle", 6), ("triangle", 9), ("full_square", 5), ("full_square", 10), ("carpet", 4), ("carpet", 5),
         ("carpet", 6), ("vicsek", 7), ("candy", 3), ("candy", 5), ("menger", 4), ("menger", 5)]


@pytest.mark.parametrize("name,r", CASES)
def test_box_generations_match_oracle(name, r):
    from paper_2110_12952_gb300 import Fractal
    fam = W.FAMILIES[name]
    g, o = Fractal.from_family(fam, r), oracle.Fractal(fam.k, fam.s, r, fam.dim, fam.table())
    rng = np.random.default_rng(r)
    x = (rng.random(o.box_cells) < 0.45).astype(np.uint8) * rng.integers(1, 256, o.box_cells).astype(np.uint8)
    rules = [W.MENGER_B5S45, W.rule_masks([4], [3, 4, 5, 26])] if fam.dim == 3 else [W.LIFE_B3S23, W.rule_masks([2, 8], [0, 1, 2, 3, 8])]
    src = torch.from_numpy(x).cuda()
    for rule, steps in zip(rules * 2, (1, 2, 3, 2)):
        whole = torch.full((o.box_cells + 64,), 77, dtype=torch.uint8, device="cuda")
        g.bb_step(src, out=whole[:o.box_cells], steps=steps, rule=rule)
        want = o.bb_step(x, rule=oracle.Rule(*rule), steps=steps)
        assert np.array_equal(whole[:o.box_cells].cpu().numpy(), want), (name, r, rule, steps)
        assert int((whole[o.box_cells:] == 77).sum()) == 64
    assert torch.equal(src.cpu(), torch.from_numpy(x))
    g.close()


def test_long_box_rows():
    # rows longer than a packing tile (16384 cells) and than a block's words: the full square at side 32768 against
    # single generations of the row kernel
    from paper_2110_12952_gb300 import Fractal
    g = Fractal.from_family(W.FULL_SQUARE, 15)
    x = torch.empty(g.box_cells, dtype=torch.uint8, device="cuda").bernoulli_(0.4)
    one = g.bb_step(g.bb_step(x, steps=1), steps=1)
    assert torch.equal(g.bb_step(x, steps=2), one)
    g.close()


@pytest.mark.parametrize("name,r,steps", [("menger", 5, 1), ("menger", 5, 3), ("carpet", 6, 2)])
def test_one_handle_on_two_streams(name, r, steps):
    # calls of one handle on streams of their own share its packed boxes; they take turns
    from paper_2110_12952_gb300 import Fractal
    g = Fractal.from_family(W.FAMILIES[name], r)
    rule = W.MENGER_B5S45 if g.dim == 3 else W.LIFE_B3S23
    x = [torch.empty(g.box_cells, dtype=torch.uint8, device="cuda").bernoulli_(p) for p in (0.2, 0.5)]
    want = [g.bb_step(v, steps=steps, rule=rule).clone() for v in x]
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    out = [[torch.empty_like(x[0]) for _ in range(6)] for _ in range(2)]
    torch.cuda.synchronize()
    for i in range(6):
        for j in range(2):
            with torch.cuda.stream(streams[j]):
                g.bb_step(x[j], out=out[j][i], steps=steps, rule=rule)
    torch.cuda.synchronize()
    assert all(torch.equal(y, want[j]) for j in range(2) for y in out[j])
    g.close()


@pytest.mark.parametrize("name,r", [("triangle", 5), ("triangle", 9), ("carpet", 5), ("carpet", 6), ("candy", 3), ("menger", 4)])
@pytest.mark.parametrize("src_off,dst_off", [(1, 0), (0, 7), (15, 9), (8, 4)])
def test_boxes_at_any_address(name, r, src_off, dst_off):
    # several generations from and to boxes that are not 16-byte aligned, called and captured after an aligned call
    from paper_2110_12952_gb300 import Fractal
    fam = W.FAMILIES[name]
    g, o = Fractal.from_family(fam, r), oracle.Fractal(fam.k, fam.s, r, fam.dim, fam.table())
    rng = np.random.default_rng(r + src_off)
    x = (rng.random(o.box_cells) < 0.45).astype(np.uint8) * rng.integers(1, 256, o.box_cells).astype(np.uint8)
    rule = W.rule_masks([4], [3, 4, 5, 26]) if fam.dim == 3 else W.rule_masks([2, 8], [0, 1, 2, 3, 8])
    whole = torch.full((o.box_cells + 64,), 77, dtype=torch.uint8, device="cuda")
    base = torch.empty(o.box_cells + 16, dtype=torch.uint8, device="cuda")
    src, dst = base[src_off:src_off + o.box_cells], whole[16 + dst_off:16 + dst_off + o.box_cells]
    src.copy_(torch.from_numpy(x))
    for captured in (False, True):
        for steps in (2, 3):
            whole.fill_(77)
            if captured:
                g.bb_step(src.clone(), steps=2, rule=rule)   # the handle's arrays
                torch.cuda.synchronize()
                graph = torch.cuda.CUDAGraph()
                with torch.cuda.graph(graph):
                    g.bb_step(src, out=dst, steps=steps, rule=rule)
                graph.replay()
                torch.cuda.synchronize()
                del graph
            else:
                g.bb_step(src, out=dst, steps=steps, rule=rule)
            want = o.bb_step(x, rule=oracle.Rule(*rule), steps=steps)
            assert np.array_equal(dst.cpu().numpy(), want), (steps, captured)
            assert int((whole == 77).sum()) == 64
    g.close()
