"""The bit-sliced step of 2D fractals (slice.cu) against the oracle, at the
sizes where its tiles, groups of 32 tiles, 32-cell chunks and 16-byte units
end: fewer tiles than a group, a last group that is not full, tiles that are
and are not whole words, one and many generations per call, rules beyond
B3/S23, buffers that are not 16-byte aligned and bytes other than 0 and 1."""
import numpy as np
import pytest
import torch

import oracle
from paper_2110_12952_gb300 import workloads as W

pytestmark = pytest.mark.gpu

RULES = [W.LIFE_B3S23, W.rule_masks([3, 6], [2, 3]), W.rule_masks([1, 8], [0, 1, 2, 5, 8])]
CASES = [("triangle", r) for r in (1, 2, 3, 5, 8, 11, 13)] + [("triangle_mirrored", 10), ("carpet", 1), ("carpet", 2),
         ("carpet", 5), ("carpet", 6), ("vicsek", 2), ("vicsek", 6), ("vicsek", 8), ("h_fractal", 3), ("h_fractal", 6),
         ("x_fractal", 7), ("chandelier", 4), ("chandelier", 8), ("candy", 2), ("candy", 5), ("empty_bottles", 6),
         ("full_square", 3), ("full_square", 9), ("cantor_set", 5), ("cantor_set", 15)]


def pair(fam, r):
    from paper_2110_12952_gb300 import Fractal
    return Fractal.from_family(fam, r), oracle.Fractal(fam.k, fam.s, r, fam.dim, fam.table())


@pytest.mark.parametrize("name,r", CASES)
def test_slice_step_matches_oracle(name, r):
    fam = W.FAMILIES[name]
    g, o = pair(fam, r)
    x = o.init_bernoulli(11 + r, 0.45)
    x[::7] *= 201   # any nonzero byte is alive
    for i, (rule, steps) in enumerate(zip(RULES * 2, (1, 2, 3, 1, 5, 8))):
        off = (0, 0, 3, 16, 9, 0)[i]
        src = torch.empty(g.cells + 64, dtype=torch.uint8, device="cuda")[off:off + g.cells]
        whole = torch.full((g.cells + 64,), 77, dtype=torch.uint8, device="cuda")
        dst = whole[64 - off - i:64 - off - i + g.cells] if i else whole[:g.cells]
        src.copy_(torch.from_numpy(x))
        g.step(src, out=dst, steps=steps, rule=rule)
        want = o.step(x, rule=oracle.Rule(*rule), steps=steps)
        assert np.array_equal(dst.cpu().numpy(), want), (name, r, rule, steps, off)
        assert int((whole == 77).sum()) == 64          # nothing written around the result
        assert np.array_equal(src.cpu().numpy(), x)
    g.check()
    g.close()


def test_slice_step_under_capture():
    # a captured call replays with new contents of the same buffers; a handle that has not run yet captures too
    fam = W.CARPET
    for warm, r in ((True, 5), (True, 7), (False, 5)):   # one block, a cooperative launch, the tile kernels
        g, o = pair(fam, r)
        x = torch.empty(g.cells, dtype=torch.uint8, device="cuda")
        y = torch.empty_like(x)
        z = torch.empty_like(x)
        if warm:
            g.step(x, out=y, steps=4)
            g.step(x, out=z, steps=1)
        else:
            assert g.tile_levels >= 0   # builds the tile kernels' tables only
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            g.step(x, out=z, steps=1)
            if warm:
                g.step(x, out=y, steps=4)
        for seed in (3, 4):
            v = o.init_bernoulli(seed, 0.5)
            x.copy_(torch.from_numpy(v))
            graph.replay()
            torch.cuda.synchronize()
            assert np.array_equal(z.cpu().numpy(), o.step(v, steps=1))
            if warm:
                assert np.array_equal(y.cpu().numpy(), o.step(v, steps=4))
        del graph
        g.close()


@pytest.mark.parametrize("name,r", [("triangle", 17), ("vicsek", 12), ("h_fractal", 10)])
def test_streamed_states_match_single_generations(name, r):
    # states too large for the resident kernel keep their packed words in memory between launches; one call of
    # several generations equals as many calls of one, and those the tile kernels'
    from paper_2110_12952_gb300 import Fractal
    fam = W.FAMILIES[name]
    g, tiles = Fractal.from_family(fam, r), Fractal.from_family(fam, r)
    tiles.tile_levels = tiles.tile_levels   # an explicit depth: the tile kernels
    x = g.init_bernoulli(5, 0.4)
    ref, one = x, x
    for steps in (1, 2, 3):
        ref = tiles.step(ref, steps=1)
        one = g.step(one, steps=1)
        assert torch.equal(one, ref)
        assert torch.equal(g.step(x, steps=steps), ref), steps
    g.check()
    g.close()
    tiles.close()


@pytest.mark.parametrize("name,r,L", [("menger", 2, 0), ("menger", 3, 0), ("menger", 4, 0), ("menger", 5, 0), ("cube", 3, 0), ("corners", 6, 0)])
def test_sliced_3d_matches_oracle(name, r, L):
    # cells with up to 19 (Menger) and 26 (the full cube) neighbours, tiles of a few and of 8000 cells
    from paper_2110_12952_gb300 import Fractal
    grid = [(x, y, z) for z in range(3) for y in range(3) for x in range(3)]
    tables = {"menger": (20, 3, W.MENGER.table()), "cube": (27, 3, np.array(grid, dtype=np.int32)),
              "corners": (4, 2, np.array([(0, 0, 0), (1, 1, 0), (1, 0, 1), (0, 1, 1)], dtype=np.int32))}
    k, s, tab = tables[name]
    g, o = Fractal(k, s, r, 3, tab), oracle.Fractal(k, s, r, 3, tab)
    x = o.init_bernoulli(r, 0.3)
    x[::7] *= 201
    rules = [W.MENGER_B5S45, W.rule_masks([4, 26], [0, 3, 4, 5, 18, 26])]
    for i, (rule, steps) in enumerate(zip(rules * 2, (2, 3, 1, 5))):
        off = (0, 3, 0, 8)[i]
        src = torch.empty(g.cells + off, dtype=torch.uint8, device="cuda")[off:]
        whole = torch.full((g.cells + 64,), 77, dtype=torch.uint8, device="cuda")
        src.copy_(torch.from_numpy(x))
        dst = whole[i:i + g.cells]
        g.step(src, out=dst, steps=steps, rule=rule)
        assert np.array_equal(dst.cpu().numpy(), o.step(x, rule=oracle.Rule(*rule), steps=steps)), (name, r, rule, steps)
        assert int((whole == 77).sum()) == 64
    g.check()
    g.close()


def test_sliced_menger_single_generations():
    # large enough for the sliced step at one generation: against the tile kernels
    from paper_2110_12952_gb300 import Fractal
    g, tiles = Fractal.from_family(W.MENGER, 6), Fractal.from_family(W.MENGER, 6)
    tiles.tile_levels = tiles.tile_levels
    x = g.init_bernoulli(5, 0.4)
    one = g.step(x, steps=1)
    assert torch.equal(one, tiles.step(x, steps=1))
    assert torch.equal(g.step(x, steps=3), tiles.step(tiles.step(one, steps=1), steps=1))
    g.close()
    tiles.close()


@pytest.mark.parametrize("name,r,steps", [("carpet", 7, 4), ("carpet", 8, 1), ("h_fractal", 8, 1), ("triangle", 16, 3), ("menger", 6, 1)])
def test_one_handle_on_two_streams(name, r, steps):
    # calls of one handle on streams of their own share its packed words; they take turns
    fam = W.FAMILIES[name]
    from paper_2110_12952_gb300 import Fractal
    g, ref = Fractal.from_family(fam, r), Fractal.from_family(fam, r)
    rule = W.MENGER_B5S45 if fam.dim == 3 else W.LIFE_B3S23
    x = [g.init_bernoulli(seed, 0.4) for seed in (1, 2)]
    want = [ref.step(v, steps=steps, rule=rule).clone() for v in x]
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    out = [[torch.empty_like(x[0]) for _ in range(6)] for _ in range(2)]
    torch.cuda.synchronize()
    for i in range(6):
        for j in range(2):
            with torch.cuda.stream(streams[j]):
                g.step(x[j], out=out[j][i], steps=steps, rule=rule)
    torch.cuda.synchronize()
    for j in range(2):
        for y in out[j]:
            assert torch.equal(y, want[j])
    g.check()
    g.close()
    ref.close()


@pytest.mark.parametrize("name,r", [("triangle", 8), ("carpet", 6), ("vicsek", 6), ("menger", 4)])
def test_sliced_call_readies_the_handle(name, r):
    # what a first step has always made possible: a captured call of another step count, the allocation-free step,
    # and a captured call once the handle has been set to the tile kernels
    fam = W.FAMILIES[name]
    g, o = pair(fam, r)
    rule = W.MENGER_B5S45 if fam.dim == 3 else W.LIFE_B3S23
    v = o.init_bernoulli(7, 0.4)
    x = torch.from_numpy(v).cuda()
    g.step(x, steps=5, rule=rule)
    want = {n: o.step(v, rule=oracle.Rule(*rule), steps=n) for n in (1, 3)}
    y = torch.empty_like(x)
    assert g._lib.fractal_step_noalloc(g._h, x.data_ptr(), y.data_ptr(), 3, rule[0], rule[1], 0) == 0
    torch.cuda.synchronize()
    assert np.array_equal(y.cpu().numpy(), want[3])
    z = torch.empty_like(x)
    for n in (1, 3, -3):
        if n < 0:
            g.tile_levels = 2
            assert g.tile_levels == 2
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            g.step(x, out=z, steps=abs(n), rule=rule)
        z.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert np.array_equal(z.cpu().numpy(), want[abs(n)]), n
        del graph
    g.check()
    g.close()


def test_several_generations_of_an_autotuned_handle():
    # the autotuner's tile depth is for single generations; calls of several go by the rules of other handles
    fam = W.FAMILIES["candy"]
    g, o = pair(fam, 4)
    v = o.init_bernoulli(9, 0.4)
    x = torch.from_numpy(v).cuda()
    g.autotune(x)
    for n in (1, 4):
        assert np.array_equal(g.step(x, steps=n).cpu().numpy(), o.step(v, steps=n))
    g.close()


@pytest.mark.parametrize("name,r,box", [("carpet", 8, False), ("h_fractal", 8, False), ("menger", 6, False), ("menger", 5, True)])
def test_single_generations_do_not_wait_for_another_stream(name, r, box):
    # a single generation on one stream is done while the same handle's earlier call on another stream has not begun
    from paper_2110_12952_gb300 import Fractal
    fam = W.FAMILIES[name]
    g, ref = Fractal.from_family(fam, r), Fractal.from_family(fam, r)
    ref.tile_levels = ref.tile_levels
    rule = W.MENGER_B5S45 if fam.dim == 3 else W.LIFE_B3S23
    one = (lambda h, v, o: h.bb_step(v, out=o, steps=1, rule=rule)) if box else (lambda h, v, o: h.step(v, out=o, steps=1, rule=rule))
    x = [ref.init_bernoulli(seed, 0.4) for seed in (1, 2)]
    if box:
        x = [ref.scatter(v) for v in x]
    out = [torch.empty_like(v) for v in x]
    for _ in range(3):
        one(g, x[0], out[0])
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    for cycles in (20_000_000, 1_000_000_000):   # (the first time loads the kernels, which may wait for the device)
        out[0].zero_()
        torch.cuda.synchronize()
        with torch.cuda.stream(a):
            torch.cuda._sleep(cycles)
            one(g, x[0], out[0])
            after = torch.cuda.Event()
            after.record()
        with torch.cuda.stream(b):
            one(g, x[1], out[1])
        b.synchronize()
        early = not after.query()
        torch.cuda.synchronize()
    assert early
    want = [ref.gather(v) for v in x] if box else x
    for v, y in zip(want, out):
        assert torch.equal(ref.gather(y) if box else y, ref.step(v, steps=1, rule=rule))
    g.check()
    g.close()
    ref.close()


GRID3 = [(x, y, z) for z in range(3) for y in range(3) for x in range(3)]


@pytest.mark.parametrize("name,r,steps", [("triangle", 11, (1,)), ("triangle", 13, (1,)), ("triangle_mirrored", 12, (1,)), ("triangle", 18, (1, 3)),
                                          ("carpet", 8, (1,)), ("h_fractal", 8, (1,)), ("h_fractal", 10, (2, 3)), ("full_square", 12, (1, 2)),
                                          ("full_square", 13, (1, 3)), ("vicsek", 12, (2, 3)), ("chandelier", 13, (1, 3)), ("x_fractal", 10, (1, 4)),
                                          ("candy", 7, (1, 2)), ("menger", 6, (1, 3)), ("cube", 5, (1, 3))])
def test_rules_and_addresses_against_the_tile_kernels(name, r, steps):
    # single generations (the single pass, packed and resident forms) and streamed states under rules without a closed
    # form, from and to buffers at odd addresses, bytes other than 0 and 1: against a handle with a tile depth of its own
    from paper_2110_12952_gb300 import Fractal
    make = (lambda: Fractal(27, 3, r, 3, np.array(GRID3, dtype=np.int32))) if name == "cube" else (lambda: Fractal.from_family(W.FAMILIES[name], r))
    g, tiles = make(), make()
    tiles.tile_levels = tiles.tile_levels
    rules = [W.rule_masks([4, 26], [0, 3, 4, 5, 18]), W.MENGER_B5S45] if g.dim == 3 else [W.rule_masks([1, 3, 8], [0, 1, 2, 5, 8]), W.LIFE_B3S23]
    x = g.init_bernoulli(3, 0.45)
    x[::7] *= 201
    base = torch.empty(g.cells + 16, dtype=torch.uint8, device="cuda")
    whole = torch.empty(g.cells + 64, dtype=torch.uint8, device="cuda")
    for rule in rules:
        want, done = x, 0
        for n in steps:
            for _ in range(n - done):
                want = tiles.step(want, steps=1, rule=rule)
            done = n
            for src_off, dst_off in ((0, 0), (0, 0), (5, 0), (0, 9), (16, 16), (1, 3)):   # (a first single generation may go to the tiles)
                src, dst = base[src_off:src_off + g.cells], whole[16 + dst_off:16 + dst_off + g.cells]
                src.copy_(x)
                whole.fill_(77)
                g.step(src, out=dst, steps=n, rule=rule)
                assert torch.equal(dst, want), (rule, n, src_off, dst_off)
                assert int((whole[:16 + dst_off] == 77).all()) and int((whole[16 + dst_off + g.cells:] == 77).all())
    g.check()
    g.close()
    tiles.close()
