"""The kernel shapes chosen by table size, and segments cut where the high word of the
Philox block index changes: the result does not depend on either.

A table that takes the large shape must give, bit for bit, what small tables over its
pieces give (they take the one-vector shape); those are checked against the oracle in
test_gpu_parity.py and, for the cuts, here."""
import ctypes

import numpy as np
import pytest

import oracle
import synthetic
from jbtest_util import check_theta, to_device, to_host, update_scale

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

F32 = np.float32
LR, DENOM, QS = float(F32(1e-3)), 3.0, 16.0


@pytest.fixture(scope="module")
def jb():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2306_10015_gb300 import build
    build.build()
    import paper_2306_10015_gb300 as pkg
    pkg.lib()
    return pkg


def pairs(K):
    seeds = [(int(m), 5, i % 3) for i, m in enumerate(synthetic.machine_ids(K, 61))]
    return seeds, synthetic.byte_codes(K, 61)


def operations(jb):
    def replay(t):
        (s1, q1), (s2, q2) = pairs(1), pairs(3)
        jb.jb_replay_updates(t, [(s1, q1, LR, DENOM), (s2, q2, LR, DENOM), (s1, q1, LR, 1.0)], QS)

    def into(t, K):
        out = [torch.zeros_like(x) for x in t.tensors]
        jb.jb_apply_updates_from(t, jb.ParamTable(out, t.flat_offsets), *pairs(K), LR, DENOM, QS)
        for x, o in zip(t.tensors, out):
            x.copy_(o)

    return {"perturb": lambda t: jb.jb_perturb(t, (7, 8, 9), 1e-3),
            "update K=1": lambda t: jb.jb_apply_updates(t, *pairs(1), LR, DENOM, QS),
            "update K=2": lambda t: jb.jb_apply_updates(t, *pairs(2), LR, DENOM, QS),
            "update K=5": lambda t: jb.jb_apply_updates(t, *pairs(5), LR, DENOM, QS),
            # too many pairs for their round keys to travel with them
            "update K=400": lambda t: jb.jb_apply_updates(t, *pairs(400), LR / 20, DENOM, QS),
            "from K=1": lambda t: into(t, 1), "from K=4": lambda t: into(t, 4), "replay": replay}


# elements of a warp tile of the large shapes: update, replay, one pair
TILES = {torch.float32: (640, 512, 512), torch.bfloat16: (768, 512, 1024)}


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("tiles,extra,shift", [(1599, 0, 0), (1600, -1, 0), (1600, 1, 0), (1700, 5, 3),
                                               (1700, 31 * 8, 0)])
def test_large_shape_equals_small_pieces(jb, dtype, tiles, extra, shift):
    for name, op in operations(jb).items():
        t = TILES[dtype][0 if name.startswith("update") and name[-1] != "1" else
                         (2 if name[-1] == "1" or name == "perturb" else 1)]
        n = tiles * t + extra
        torch.manual_seed(n)
        base = torch.randn(n + 16, device="cuda").mul_(0.02).to(dtype)
        whole, parts = base.clone(), base.clone()
        op(jb.ParamTable([whole[shift:shift + n]], [11]))
        cuts = [0, 1, 9, 4099] + list(range(300_001, n, 300_001)) + [n - 3, n]
        for a, b in zip(cuts, cuts[1:]):
            op(jb.ParamTable([parts[shift + a:shift + b]], [11 + a]))
        torch.cuda.synchronize()
        assert torch.equal(whole.view(torch.uint8), parts.view(torch.uint8)), name


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("count,largest,first", [(1700, 9, 3), (5000, 300, 0), (2500, 900, 5)])
def test_thousands_of_tiny_tensors(jb, dtype, count, largest, first):
    """Tables that take the large shape by their number of tensors, with tiles that are mostly
    empty, in several launches, against one tensor over all of them."""
    rng = np.random.default_rng(count)
    ends = np.cumsum(rng.integers(1, largest + 1, count)).tolist()
    spans = list(zip([0] + ends, ends))
    n = ends[-1]
    torch.manual_seed(count)
    base = torch.randn(n, device="cuda").mul_(0.02).to(dtype)
    for name, op in operations(jb).items():
        whole, parts = base.clone(), base.clone()
        op(jb.ParamTable([whole], [first]))
        op(jb.ParamTable([parts[a:b] for a, b in spans], [first + a for a, _ in spans]))
        assert torch.equal(whole.view(torch.uint8), parts.view(torch.uint8)), name
    sums = [torch.zeros(1, dtype=torch.int64, device="cuda") for _ in range(2)]
    starts = sorted({min((a + 7) // 8 * 8, n) for a, _ in spans} | {n})  # a window belongs to one tensor
    cuts = list(zip(starts, starts[1:]))
    jb.jb_checksum(jb.ParamTable([base], [8]), sums[0])
    jb.jb_checksum(jb.ParamTable([base[a:b] for a, b in cuts], [8 + a for a, _ in cuts]), sums[1])
    assert sums[0].item() == sums[1].item()


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("n", [7, 33, 4099, 400_003, 1_700_021])
def test_off_grid_equals_aligned(jb, dtype, n):
    """Tensors that start at every element of the 16-byte grid of their flat offsets (8, 4
    and 2 byte alignment, a head or none) against the aligned one; what lies around them
    stays as it was. From a source and into a destination of other alignments too."""
    torch.manual_seed(n)
    values = torch.randn(n, device="cuda").mul_(0.02).to(dtype)
    per = 16 // values.element_size()

    def placed(shift, fill=7.0):
        buf = torch.full((n + 64,), fill, device="cuda", dtype=dtype)
        buf[16 + shift:16 + shift + n] = values
        return buf, buf[16 + shift:16 + shift + n]

    def check(buf, part, want, what):
        assert torch.equal(part.view(torch.uint8), want.view(torch.uint8)), what
        start = part.storage_offset()
        assert bool((buf[:start] == 7.0).all()) and bool((buf[start + n:] == 7.0).all()), what

    ops = operations(jb)
    for fo in (8, 11):
        wants = {}
        for name, op in ops.items():
            buf, part = placed(fo % per)  # on the grid
            op(jb.ParamTable([part], [fo]))
            wants[name] = part.clone()
        total = torch.zeros(1, dtype=torch.int64, device="cuda")
        jb.jb_checksum(jb.ParamTable([placed(fo % per)[1]], [fo]), total)
        for shift in range(per):
            for name, op in ops.items():
                if name.startswith("from"):
                    continue
                buf, part = placed(shift)
                op(jb.ParamTable([part], [fo]))
                check(buf, part, wants[name], (fo, shift, name))
            buf, part = placed(shift)
            got = torch.zeros(1, dtype=torch.int64, device="cuda")
            jb.jb_checksum(jb.ParamTable([part], [fo]), got)
            assert int(got.item()) == int(total.item())
            for K in (1, 4):
                for to in (0, 1, 2, per // 2):
                    src, s = placed(shift)
                    dst, d = placed(to)
                    d.zero_()
                    jb.jb_apply_updates_from(jb.ParamTable([s], [fo]), jb.ParamTable([d], [fo]), *pairs(K), LR,
                                             DENOM, QS, write_src=(to == 1))
                    check(dst, d, wants[f"from K={K}"], (fo, shift, to, K))
                    check(src, s, wants[f"from K={K}"] if to == 1 else values, (fo, shift, to, K))


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("K", [2, 3, 8, 33, 100])
def test_pairs_shared_out(jb, dtype, K):
    """Tables of few tiles, whose pairs are shared out among warps, against one table over
    all of them, which is too large for that: in place, from a source, and a replay whose
    groups end inside a chunk of pairs. The piece lengths give groups of 16, 8 and 4 warps."""
    seeds, q = pairs(K)
    steps = [(seeds[a:b], q[a:b], LR, 1.0 + a) for a, b in zip([0, 1, K // 2], [1, max(K // 2, 1), K]) if b > a]

    def into(t, refresh):
        out = [torch.zeros_like(x) for x in t.tensors]
        jb.jb_apply_updates_from(t, jb.ParamTable(out, t.flat_offsets), seeds, q, LR, DENOM, QS,
                                 write_src=refresh)
        if not refresh:
            for x, o in zip(t.tensors, out):
                x.copy_(o)

    for op in (lambda t: jb.jb_apply_updates(t, seeds, q, LR, DENOM, QS), lambda t: into(t, False),
               lambda t: into(t, True), lambda t: jb.jb_replay_updates(t, steps, QS)):
        torch.manual_seed(K)
        n = 400_003
        base = torch.randn(n, device="cuda").mul_(0.02).to(dtype)
        whole, parts = base.clone(), base.clone()
        op(jb.ParamTable([whole], [6]))
        cuts = np.cumsum([0, 1, 2, 3, 122, 128, 129, 5003, 152 * 128, 152 * 128 + 1, 304 * 128 + 7, 70_001, 77_000])
        cuts = list(cuts) + [n - 70_000, n]
        for a, b in zip(cuts, cuts[1:]):
            mid = (a + b) // 2
            tensors = [parts[a:b]] if b - a < 1000 else [parts[a:mid], parts[mid:b]]
            op(jb.ParamTable(tensors, [6 + a, 6 + mid][:len(tensors)]))
        torch.cuda.synchronize()
        assert torch.equal(whole.view(torch.uint8), parts.view(torch.uint8))


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("vectors", [1, 31 * 32 + 1, 32 * 32, 32 * 32 + 1, 1600 * 192 - 1, 1600 * 192 + 33])
def test_checksum_shapes(jb, dtype, vectors):
    """One CTA that stores its sum, several that add to a cleared one, the large shape."""
    per = 4 if dtype == "f32" else 8
    for n, fo in ((vectors * per, 0), (vectors * per - 1, 5), (vectors * per, (1 << 33) - 8)):
        v = synthetic.normal_values(n, 0.02, 64)
        v = v if dtype == "f32" else oracle.round_bf16(v.astype(np.float64))
        out = torch.full((1,), 12345, dtype=torch.int64, device="cuda")
        jb.jb_checksum(jb.ParamTable([to_device(v)], [fo]), out)
        assert int(out.item()) & (2**64 - 1) == oracle.checksum([v], [fo])


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("boundary", [1 << 33, 1 << 34, 3 << 33])
def test_segment_across_a_cut(jb, dtype, boundary):
    """A segment that crosses a multiple of 2^33 elements (2^34: another high word)."""
    for before, K in ((1001, 3), (1, 1), (4096, 2)):
        v = synthetic.normal_values(5003, 0.02, 62)
        v = v if dtype == "f32" else oracle.round_bf16(v.astype(np.float64))
        fo = boundary - before
        dev = to_device(v)
        seeds, q = pairs(K)
        jb.jb_apply_updates(jb.ParamTable([dev], [fo]), seeds, q, LR, DENOM, QS)
        torch.cuda.synchronize()
        scale = update_scale(v, np.arange(fo, fo + v.size, dtype=np.uint64), seeds, q, LR, DENOM, QS)
        check_theta(to_host(dev), oracle.update(v, fo, seeds, q, LR, DENOM, QS), scale, f"{boundary}")


def kernels_of(call):
    """How many kernels a call launches: the kernel nodes of a graph captured from it."""
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        call()
    cu, raw, n = ctypes.CDLL("libcuda.so.1"), ctypes.c_void_p(graph.raw_cuda_graph()), ctypes.c_size_t()
    assert cu.cuGraphGetNodes(raw, None, ctypes.byref(n)) == 0
    nodes = (ctypes.c_void_p * n.value)()
    assert cu.cuGraphGetNodes(raw, nodes, ctypes.byref(n)) == 0
    kinds = [ctypes.c_int(-1) for _ in range(n.value)]
    for node, kind in zip(nodes, kinds):
        assert cu.cuGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(kind)) == 0
    return sum(kind.value == 0 for kind in kinds)


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("boundary", [1 << 34, 3 << 34, 1 << 35])
@pytest.mark.parametrize("shift,parts", [(0, 1), (0, 7), (1, 7)])
def test_large_table_across_a_high_word(jb, dtype, boundary, shift, parts):
    """Tables of the large shape whose indices have two high words take one launch if they fit
    it, and give what the pieces on either side of the boundary give by themselves: one tensor
    that crosses, several, in any order (a third run of high words is another launch), on the
    grid and off it."""
    ops = operations(jb)
    ops["update K=512"] = lambda t: jb.jb_apply_updates(t, *pairs(512), LR / 20, DENOM, QS)  # two sets do not fit

    def refresh(t, K):
        out = [torch.zeros_like(x) for x in t.tensors]
        jb.jb_apply_updates_from(t, jb.ParamTable(out, t.flat_offsets), *pairs(K), LR, DENOM, QS, write_src=True)
        assert all(torch.equal(x.view(torch.uint8), o.view(torch.uint8)) for x, o in zip(t.tensors, out))

    ops["refresh K=1"], ops["refresh K=4"] = (lambda t: refresh(t, 1)), (lambda t: refresh(t, 4))
    n, before = 3_000_003, 1_400_008
    torch.manual_seed(parts)
    base = torch.randn(n + 16, device="cuda").mul_(0.02).to(dtype)
    ends = [n * (i + 1) // parts for i in range(parts)]
    spans = list(zip([0] + ends, ends))
    orders = {"in order": spans, "reversed": spans[::-1], "three runs": spans[1:] + spans[:1]}
    for name, op in ops.items():
        want = base.clone()
        for a, b in ((0, before), (before, n)):
            op(jb.ParamTable([want[shift + a:shift + b]], [boundary - before + a]))
        for what, order in orders.items():
            got = base.clone()
            op(jb.ParamTable([got[shift + a:shift + b] for a, b in order], [boundary - before + a for a, _ in order]))
            assert torch.equal(got.view(torch.uint8), want.view(torch.uint8)), (name, what)

    def checksum(spans):
        out = torch.zeros(1, dtype=torch.int64, device="cuda")
        jb.jb_checksum(jb.ParamTable([base[shift + a:shift + b] for a, b in spans],
                                     [boundary - before + a for a, _ in spans]), out)
        return int(out.item()) & (2**64 - 1)

    for spans in orders.values():
        alone = sum(checksum([(a, b)] if b <= before or a >= before else [(a, before)]) +
                    (checksum([(before, b)]) if a < before < b else 0) for a, b in spans)
        assert checksum(spans) == alone % 2**64

    table = jb.ParamTable([base[shift + a:shift + b] for a, b in orders["in order"]],
                          [boundary - before + a for a, _ in orders["in order"]])
    total = torch.zeros(1, dtype=torch.int64, device="cuda")
    for call in (lambda: jb.jb_perturb(table, (7, 8, 9), 1e-3), lambda: jb.jb_apply_updates(table, *pairs(5), LR, DENOM, QS),
                 lambda: jb.jb_replay_updates(table, [(*pairs(2), LR, 1.0), (*pairs(1), LR, 1.0)], QS),
                 lambda: jb.jb_checksum(table, total)):
        assert kernels_of(call) == 1


def test_q4_across_a_high_word(jb):
    """4-bit tensors whose Philox block indices cross 2^32, or lie above it."""
    n = 64 * 40 + 33
    for fos in ([(1 << 34) - 1028], [1 << 34], [64, (1 << 35) + 8]):
        host, dev = [], []
        for i, _ in enumerate(fos):
            codes, scale = oracle.q4_quantize(synthetic.normal_values(n, 0.02, 63 + i).astype(np.float64))
            host.append((codes, scale))
            pad = np.zeros(codes.size + 16, dtype=np.uint8)
            pad[:codes.size] = codes
            dev.append((torch.from_numpy(pad).cuda(), torch.from_numpy(scale.copy()).cuda(), n))
        jb.jb_perturb_q4(jb.Q4Table(dev, fos), (3, 4, 5), 1e-3)
        torch.cuda.synchronize()
        level = jb.jb_q4_levels().astype(np.float64)
        for (codes, scale), (dc, ds, _), fo in zip(host, dev, fos):
            old = np.empty(2 * codes.size, dtype=np.int64)
            old[0::2], old[1::2] = codes & 15, codes >> 4
            w = level[old[:n]] * np.repeat(scale, 64)[:n].astype(np.float64)
            w += float(F32(1e-3)) * oracle.gaussian_range((3, 4, 5), fo, n)
            want = np.abs(np.pad(w, (0, 64 * scale.size - n))).reshape(-1, 64).max(1)
            # w' is one fp32 multiply-add of values below 0.2 with z to 1e-6
            assert np.all(np.abs(ds.cpu().numpy() - want) <= 2e-8 + 1e-9)
            new = dc.cpu().numpy()[:codes.size].astype(np.int64)
            got = np.empty(2 * codes.size, dtype=np.int64)
            got[0::2], got[1::2] = new & 15, new >> 4
            near = np.abs((w / np.repeat(want, 64)[:n])[:, None] - level[None, :]).argmin(1)
            # ties within fp32 error of a midpoint: none expected among 2593 weights
            assert np.count_nonzero(got[:n] != near) <= 1
