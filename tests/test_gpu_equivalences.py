"""Randomised equivalences between the library's entry points, all on the GPU: the shard-by-shard
forms against the all-shard call, ws_pack_sets against ws_pack, the fused route against the
separate kernels, and one kernel per replica over R weight lists against the unpacked gathered
buffer - over random tensor lists (also more than 1024 tensors), shard counts up to 1024,
alignments, tile sizes, layouts, optimizers and dtypes.  Bit for bit, except where a shard's slices
are less aligned than the whole buffers (the norm-based optimizers then sum in another order)."""
import numpy as np
import pytest
import torch

from paper_2004_13336_b200 import binding as B
from paper_2004_13336_b200 import workloads as W
from tests._util import TOL_FP32

pytestmark = pytest.mark.gpu
DEV = "cuda"
POOL = [0, 1, 2, 5, 8, 31, 32, 33, 100, 255, 256, 1000, 1024, 1025, 2048, 4097, 9001, 30011, 70001]


@pytest.mark.parametrize("case", range(40))
def test_entry_points_agree(case):
    rng = np.random.default_rng(9000 + case)
    big_T = case % 13 == 5
    T = int(rng.integers(1030, 1200)) if big_T else int(rng.integers(1, 16))
    numel = [int(x) for x in rng.choice(POOL[:8] if big_T else POOL, T)]
    if sum(numel) == 0:
        numel[0] = 40
    R = int(rng.choice([1, 3, 8] if big_T else [1, 2, 3, 4, 7, 8, 12, 33, 100]))
    if case % 13 == 9:
        R, numel = int(rng.choice([257, 600, 1024])), numel[:4]
        if sum(numel) == 0:
            numel[0] = 40
    shapes = [(k,) for k in numel]
    A, tile = int(rng.choice([8, 16, 32, 128])), int(rng.choice([0, 1024, 2048]))
    layout = str(rng.choice(["per_tensor", "concat"]))
    opt = str(rng.choice(["sgdm", "adam", "lamb", "lars"]))
    gdt = torch.bfloat16 if rng.random() < 0.4 else torch.float32
    odt = torch.bfloat16 if rng.random() < 0.4 else torch.float32
    wl = W.Workload("f", shapes, R=R, opt=opt, hyper={}, grad_dtype=gdt, grad_std=1e-3, seed=case)
    h = dict(lr=1e-3, beta1=0.9, beta2=0.999, eps=1e-8, weight_decay=0.0, momentum=0.0, grad_scale=1.0,
             step=int(rng.integers(1, 20)))
    if opt == "sgdm":
        h.update(lr=0.1, momentum=0.9, weight_decay=5e-5)
    if opt == "lamb":
        h.update(eps=1e-6, weight_decay=0.01)
    if opt == "lars":
        h.update(lr=10.0, momentum=0.9, weight_decay=5e-5, trust_coeff=0.001)
    hy = B.make_hyper(opt, h)
    w, m, v = W.make_state(wl, DEV)
    g = W.make_grads(wl, DEV)
    plan = B.Plan(shapes, R, A, tile, layout=layout)
    S, G = plan.S, plan.G
    has_v = opt in ("adam", "lamb")
    norm_based = opt in ("lamb", "lars")

    def packed(lst, dt=torch.float32):
        b = torch.full((G,), float("nan"), dtype=dt, device=DEV)
        B.ws_pack(plan, lst, b)
        return b
    pw, pm, pv = packed(w), packed(m), packed(v)
    pg = [packed(gk, gdt) for gk in g]
    bits = torch.int16 if gdt == torch.bfloat16 else torch.int32
    many = [torch.full((G,), float("nan"), dtype=gdt, device=DEV) for _ in range(R)]
    B.ws_pack_sets(plan, B.TensorTable(plan, g), many)
    for a, b in zip(pg, many):
        assert torch.equal(a.view(bits), b.view(bits)), "ws_pack_sets"

    aw, am, av = pw.clone(), pm.clone(), pv.clone()
    ws = torch.full((max(16, plan.workspace_bytes(opt)),), 0xFF, dtype=torch.uint8, device=DEV)
    ga = torch.full((G,), 5.0, dtype=odt, device=DEV)
    B.ws_shard_update(plan, -1, pg, aw, am, av if has_v else None, hy, ga, ws)
    assert bool(torch.isfinite(aw).all())

    bw, bm, bv = pw.clone(), pm.clone(), pv.clone()
    gb = torch.full((G,), 5.0, dtype=odt, device=DEV)
    ws2 = torch.full_like(ws, 0xFF)
    sm = int(rng.integers(2))
    sl = [slice(r * S, (r + 1) * S) for r in range(R)]
    gr = (lambda r: [b[sl[r]] for b in pg]) if sm else (lambda r: pg)
    if not norm_based:
        for r in range(R):
            B.ws_shard_update(plan, r, gr(r), bw[sl[r]], bm[sl[r]], bv[sl[r]] if has_v else None, hy, gb, None,
                              slice_mode=sm)
    else:
        for r in range(R):
            if opt == "lamb":
                B.ws_lamb_partial(plan, r, gr(r), bw[sl[r]], bm[sl[r]], bv[sl[r]], hy, ws2, slice_mode=sm)
            else:
                B.ws_lars_partial(plan, r, gr(r), bw[sl[r]], bm[sl[r]], hy, ws2, slice_mode=sm)
        if opt == "lamb":
            B.ws_lamb_finalize(plan, ws2)
        else:
            B.ws_lars_finalize(plan, hy, ws2)
        for r in range(R):
            if opt == "lamb":
                B.ws_lamb_apply(plan, r, bw[sl[r]], bm[sl[r]], bv[sl[r]], hy, ws2, gb)
            else:
                B.ws_lars_apply(plan, r, bw[sl[r]], bm[sl[r]], hy, ws2, gb)
    for x, y, nm in ((aw, bw, "w"), (am, bm, "m"), (av, bv, "v"), (ga, gb, "gathered")):
        if nm == "v" and not has_v:
            continue
        if norm_based:
            assert torch.allclose(x.float(), y.float(), rtol=1e-2 if nm == "gathered" else 2e-5, atol=1e-7), nm
        else:
            assert torch.equal(x, y), nm

    fw, fm, fv = pw.clone(), pm.clone(), pv.clone()
    outs = [torch.full((k,), 9.0, dtype=odt, device=DEV) for k in numel]
    B.ws_fused_update(plan, -1, B.TensorTable(plan, g), fw, fm, fv if has_v else None, hy,
                      B.TensorTable(plan, [outs]), torch.full_like(ws, 0xFF))
    ref = [torch.full((k,), 7.0, dtype=odt, device=DEV) for k in numel]
    B.ws_unpack(plan, ga, ref)
    assert torch.equal(fw, aw) and torch.equal(fm, am), "fused state"
    for a, b in zip(outs, ref):
        assert torch.equal(a, b), "fused weights"

    if not norm_based and R <= 16:
        lists = [[torch.full((k,), 9.0, dtype=odt, device=DEV) for k in numel] for _ in range(R)]
        rw, rm, rv = pw.clone(), pm.clone(), pv.clone()
        gt, wt = B.TensorTable(plan, g), B.TensorTable(plan, lists)
        for r in range(R):
            B.ws_fused_update(plan, r, gt, rw[sl[r]], rm[sl[r]], rv[sl[r]] if has_v else None, hy, wt, None)
        assert torch.equal(rw, aw), "replica kernels: state"
        for k in range(R):
            for a, b in zip(lists[k], ref):
                assert torch.equal(a, b), "replica kernels: weights"


@pytest.mark.parametrize("layout", ["per_tensor", "concat"])
@pytest.mark.parametrize("gdtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("opt", ["sgdm", "adam"])
@pytest.mark.parametrize("R", [33, 64, 128, 129, 257, 1024])
def test_many_copies_one_thread_or_a_group_per_warp(R, opt, gdtype, layout):
    # one shard's slices (small: the groups of copies go to the warps of a CTA) against the same sums in one thread per
    # element (the formatting-fused form): a last block, a last group and a last vector that are not full, shards of
    # padding only; the sums against 64 bits
    shapes = [(1031,), (3,), (257, 9), (0,), (128,), (41, 100)]
    numel = [int(np.prod(s)) for s in shapes]
    M = 3
    plan = B.Plan(shapes, M, 8, layout=layout)
    gen = torch.Generator(device=DEV).manual_seed(R)
    def draw(std):
        return [torch.randn(n, generator=gen, device=DEV) * std for n in numel]
    w, m, v = draw(0.02), draw(1e-3), [x.abs() for x in draw(1e-5)]
    g = [[x.to(gdtype) for x in draw(1e-3)] for _ in range(R)]
    hy = B.make_hyper(opt, dict(lr=1.0 if opt == "sgdm" else 1e-3, beta1=0.9, beta2=0.999, eps=1e-8, weight_decay=0.0,
                                momentum=0.0, grad_scale=1.0, step=3))

    def packed(lst, dt=torch.float32):
        b = torch.full((plan.G,), float("nan"), dtype=dt, device=DEV)
        B.ws_pack(plan, lst, b)
        return b

    state = [packed(x) for x in (w, m, v)]
    if opt == "sgdm":
        state[2] = None
    one = [None if x is None else x.clone() for x in state]
    wt = [torch.empty(n, device=DEV) for n in numel]
    B.ws_fused_update(plan, -1, B.TensorTable(plan, g), *one, hy, B.TensorTable(plan, [wt]))
    pg = [packed(x, gdtype) for x in g]
    S = plan.S
    gathered = torch.full((plan.G,), 7.0, dtype=torch.bfloat16, device=DEV)
    for r in range(M):
        cut = [None if x is None else x[r * S:(r + 1) * S].clone() for x in state]
        B.ws_shard_update(plan, r, [x[r * S:(r + 1) * S].clone() for x in pg], *cut, hy, gathered, None, slice_mode=1)
        for a, b in zip(cut, one):
            assert a is None or torch.equal(a, b[r * S:(r + 1) * S])
    assert torch.equal(gathered, one[0].to(torch.bfloat16))
    if opt == "sgdm":                              # m' is the sum itself: two roundings of compensated sums of trees of 16
        for t, n in enumerate(numel):
            exact = sum(gk[t].double() for gk in g)
            lst = [torch.empty(k, device=DEV) for k in numel]
            B.ws_unpack(plan, one[1], lst)
            got = lst[t].double()
            # a tree of 16 has 4 levels, each at most 2^-24 of its partial sums, which 16 sum |g| / R bound
            bound = 6 * 2.0 ** -24 * sum(gk[t].double().abs() for gk in g)
            assert bool(((got - exact).abs() <= bound).all())


@pytest.mark.parametrize("gdtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("S,form", [(2048, "slices"), (1 << 19, "slices"), (2048, "fused")])   # a group per warp, one thread, one thread
@pytest.mark.parametrize("R", [129, 250, 256])       # a last group of one copy, of two blocks (the last not full), of two full ones
def test_an_infinite_copy_among_many(R, S, form, gdtype):
    # in the last tree block it leaves the sum +-inf, elsewhere nothing finite, and no other element changes
    plan = B.Plan([(S,)], 1, 8)
    gen = torch.Generator(device=DEV).manual_seed(R)
    g = [(torch.randn(S, generator=gen, device=DEV) * 1e-3).to(gdtype) for _ in range(R)]
    hy = B.make_hyper("sgdm", dict(lr=0.0, beta1=0.9, beta2=0.999, eps=1e-8, weight_decay=0.0, momentum=0.0, grad_scale=1.0, step=1))

    def summed():                                    # m' without momentum and decay is the sum
        w, m = torch.zeros(S, device=DEV), torch.zeros(S, device=DEV)
        if form == "slices":
            B.ws_shard_update(plan, 0, g, w, m, None, hy, slice_mode=1)
        else:
            B.ws_fused_update(plan, -1, B.TensorTable(plan, [[x] for x in g]), None, m, None, hy, B.TensorTable(plan, [[w]]))
        return m

    clean = summed()
    inf = float("inf")
    last = (R - 1) // 16 * 16
    placed = {3: (R - 1, inf), 4: (R - 1, -inf), 5: (last, inf), 701: (last, -inf), 900: (0, inf), 901: (40, -inf)}
    for e, (k, x) in placed.items():
        g[k][e] = x
    got = summed()
    for e, (k, x) in placed.items():
        if k >= last:
            assert got[e].item() == x, e
        assert not torch.isfinite(got[e]), e
    rest = torch.ones(S, dtype=torch.bool, device=DEV)
    rest[list(placed)] = False
    assert torch.isfinite(clean).all() and torch.equal(got[rest], clean[rest])


@pytest.mark.parametrize("layout", ["per_tensor", "concat"])
@pytest.mark.parametrize("opt", ["lamb", "lars"])
@pytest.mark.parametrize("R,items", [(1, "few"), (3, "few"), (1, "some"), (3, "some"), (3, "many")])
def test_ratios_formed_in_phase_two(R, items, opt, layout):
    # small models form the ratios in phase 2 ("few" and, with other registers, "some"), larger ones in a launch of their own: ratios and norms (also those
    # of a tensor without elements), state and weights are bit for bit those of the calls shard by shard
    shapes = [(0,), (257, 33), (1,), (0, 5), (40, 1031), (64,), (0,)] + {"few": [], "some": [(490, 1000)], "many": [(700, 3000)]}[items]
    wl = W.Workload("f", shapes, R=R, opt=opt, hyper={}, grad_dtype=torch.float32, grad_std=1e-3, seed=R)
    plan = B.Plan(shapes, R, 32, 1024, layout=layout, one_launch=False)
    n = plan.ntiles * (R if layout == "per_tensor" else 1)
    assert {"few": n <= 444, "some": 444 < n <= 592, "many": n > 592}[items]
    h = dict(lr=1e-3, beta1=0.9, beta2=0.999, eps=1e-6, weight_decay=0.01, momentum=0.9, grad_scale=1.0, step=4, trust_coeff=0.001)
    hy = B.make_hyper(opt, h)
    w, m, v = W.make_state(wl, DEV)
    g = W.make_grads(wl, DEV)

    def packed(lst):
        b = torch.empty(plan.G, device=DEV)
        B.ws_pack(plan, lst, b)
        return b

    state = [packed(w), packed(m), packed(v) if opt == "lamb" else None]
    pg = [packed(x) for x in g]
    per = [None if x is None else x.clone() for x in state]
    one, fused = ([None if x is None else x.clone() for x in state] for _ in range(2))
    wsp, wso, wsf = (torch.full((plan.workspace_bytes(opt),), x, dtype=torch.uint8, device=DEV) for x in (0, 0xA5, 0x5A))
    go, gp = (torch.zeros(plan.G, dtype=torch.bfloat16, device=DEV) for _ in range(2))
    B.ws_shard_update(plan, -1, pg, *one, hy, go, wso)
    cut = lambda r: [None if x is None else x[r * plan.S:(r + 1) * plan.S] for x in per]  # noqa: E731
    for r in range(R):
        sw, sm, sv = cut(r)
        B.ws_lamb_partial(plan, r, pg, sw, sm, sv, hy, wsp) if opt == "lamb" else B.ws_lars_partial(plan, r, pg, sw, sm, hy, wsp)
    B.ws_lamb_finalize(plan, wsp) if opt == "lamb" else B.ws_lars_finalize(plan, hy, wsp)
    for r in range(R):
        sw, sm, sv = cut(r)
        B.ws_lamb_apply(plan, r, sw, sm, sv, hy, wsp, gp) if opt == "lamb" else B.ws_lars_apply(plan, r, sw, sm, hy, wsp, gp)
    wt = [torch.zeros(x.numel(), device=DEV) for x in w]
    B.ws_fused_update(plan, -1, B.TensorTable(plan, g), *fused, hy, B.TensorTable(plan, [wt]), wsf)
    head = (4 * plan.T + 15) // 16 * 16 + 16 * plan.T           # ratios and squared norms
    off = plan.sync_status_offset()
    for ws, st in ((wso, one), (wsf, fused)):
        assert torch.equal(ws[:4 * plan.T], wsp[:4 * plan.T]) and torch.equal(ws[head - 16 * plan.T:head], wsp[head - 16 * plan.T:head])
        assert int(ws[off:off + 4].view(torch.int32).item()) == 0
        assert all(a is None or torch.equal(a, b) for a, b in zip(st, per))
    assert torch.equal(go, gp)


@pytest.mark.parametrize("gdtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("tile", [1 << 15, 1 << 17, 1 << 20])
def test_few_long_tiles_among_short_ones(tile, gdtype):
    # the average tile is short, the longest is not: packed buffers, state and weights are those of a plan with tiles of 1024
    numel, R = [40] * 2500 + [700_001] + [17] * 100, 2
    got = []
    for t in (1024, tile):
        plan = B.Plan([(n,) for n in numel], R, 8, t)
        gen = torch.Generator(device=DEV).manual_seed(3)
        offs = [plan.arena_offsets()[i] for i in range(plan.T)]
        arena = lambda std, dt=torch.float32: (torch.randn(plan.arena_elems, generator=gen, device=DEV) * std).to(dt)  # noqa: E731,B023
        views = lambda x: [x[o:o + n] for o, n in zip(offs, numel)]  # noqa: E731,B023
        w, g = arena(0.02), [arena(1e-3, gdtype) for _ in range(R)]
        m, v = torch.zeros(plan.G, device=DEV), torch.zeros(plan.G, device=DEV)
        packed = [torch.empty(plan.G, dtype=gdtype, device=DEV) for _ in range(R)]
        table = B.TensorTable(plan, [views(x) for x in g])
        B.ws_pack_sets(plan, table, packed)
        hy = B.make_hyper("adam", dict(lr=1e-3, beta1=0.9, beta2=0.999, eps=1e-8, weight_decay=0.0, momentum=0.0, grad_scale=1.0, step=1))
        B.ws_fused_update(plan, -1, table, None, m, v, hy, B.TensorTable(plan, [views(w)]))
        flat, back = torch.empty(plan.G, device=DEV), torch.zeros_like(w)
        B.ws_pack(plan, views(w), flat)
        B.ws_unpack(plan, flat, views(back))
        assert all(torch.equal(a, b) for a, b in zip(views(w), views(back)))
        got.append([w, m, v, flat] + packed)
    assert all(torch.equal(a, b) for a, b in zip(*got))


@pytest.mark.parametrize("gdtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("shards,copies,align,layout,shift", [(3, 3, 8, "per_tensor", 0), (8, 8, 8, "per_tensor", 16), (8, 12, 32, "concat", 16),
                                                              (12, 4, 32, "per_tensor", 0), (5000, 2, 8, "concat", 0), (5000, 16, 32, "concat", 0),
                                                              (5000, 1, 32, "concat", 16), (16, 32, 32, "per_tensor", 16), (32, 32, 8, "per_tensor", 0)])
def test_many_short_tiles(shards, copies, align, layout, shift, gdtype):
    # 1200 tensors of 0 to 900 elements (two tables of tensor pointers) cut into shards: pieces of 8 to a few hundred
    # elements, where pack and unpack give a warp to a tile and an update has CTAs of 64 or 128 threads; tensors on
    # 32-byte boundaries, or 16 bytes beside one (`shift`), and with `align` 32 vectors of 32 bytes in bf16 too
    rng = np.random.default_rng(shards + align)
    numel = [int(x) for x in rng.integers(0, 900, 1200)] + [1, 7, 8, 9, 1024, 2049]
    plan = B.Plan([(n,) for n in numel], shards, align, layout=layout)
    assert plan.ntiles * (1 if layout == "concat" else shards) > 444
    gen = torch.Generator(device=DEV).manual_seed(shards + copies)
    offs, at = [], 0
    for n in numel:
        offs.append(at)
        at += (n + 15) // 16 * 16 + 16

    def arena(std, dt=torch.float32):
        return (torch.randn(at + 16, generator=gen, device=DEV) * std).to(dt)

    def views(t, size=None):
        k = shift // (size or t.element_size())
        return [t[o + k:o + k + n] for o, n in zip(offs, numel)]

    def placed(lst):                                # [R][S] by the definition of the layout
        flat = torch.zeros(plan.G, dtype=lst[0].dtype, device=DEV)
        for s, x in zip(plan.segments(), lst):
            if x.numel() == 0:
                continue
            if layout == "concat":
                flat[s.shard_off:s.shard_off + x.numel()] = x
            else:
                full = torch.zeros(shards * s.piece, dtype=x.dtype, device=DEV)
                full[:x.numel()] = x
                flat.view(shards, plan.S)[:, s.shard_off:s.shard_off + s.piece] = full.view(shards, s.piece)
        return flat

    w, m, v, g = arena(0.02), arena(1e-3), arena(1e-5).abs(), [arena(1e-3, gdtype) for _ in range(copies)]
    state = []
    for t in (w, m, v, g[0]):
        flat = torch.full((plan.G,), float("nan"), dtype=t.dtype, device=DEV)
        B.ws_pack(plan, views(t), flat)
        assert torch.equal(flat, placed(views(t)))
        back, expect = torch.full_like(t, 7.0), torch.full_like(t, 7.0)
        B.ws_unpack(plan, flat, views(back))
        for a, b in zip(views(expect), views(t)):
            a.copy_(b)
        assert torch.equal(back, expect)            # (and nothing between the tensors)
        state.append(flat)
    packed = [torch.full((plan.G,), float("nan"), dtype=gdtype, device=DEV) for _ in range(copies)]
    table = B.TensorTable(plan, [views(t) for t in g])
    B.ws_pack_sets(plan, table, packed)
    assert all(torch.equal(a, placed(views(b))) for a, b in zip(packed, g))

    def close(x, ref):
        # a chain of fewer than 16 fp32 roundings of 2^-24 (tree, compensated sum, moments, root, quotient) is below 1e-6 of
        # the operands' scale, the measure that every output of these optimizers is held to
        rms = ref.square().mean().sqrt()
        return bool(((x.double() - ref).abs() <= TOL_FP32 * torch.maximum(ref.abs(), rms)).all())

    # both elementwise optimizers against 64 bits; several weight lists, the packed form and the master form against the first
    gs = sum(t.double() for t in g).roll(shift // 4 - shift // g[0].element_size())      # at the places of the fp32 tensors
    for opt in ("adam", "sgdm"):
        hy = B.make_hyper(opt, dict(lr=1e-3, beta1=0.9, beta2=0.999, eps=1e-8, weight_decay=0.0, momentum=0.9, grad_scale=1.0, step=10))
        s = [x.clone() for x in state[:3]]
        outs = [torch.zeros_like(w) for _ in range(min(copies, 3))]
        B.ws_fused_update(plan, -1, table, *s, hy, B.TensorTable(plan, [views(x) for x in outs]))
        if opt == "adam":
            m1, v1 = 0.9 * m.double() + 0.1 * gs, 0.999 * v.double() + 0.001 * gs * gs
            w1 = w.double() - 1e-3 * (m1 / (1 - 0.9 ** 10)) / ((v1 / (1 - 0.999 ** 10)).sqrt() + 1e-8)
        else:
            m1, v1 = 0.9 * m.double() + gs, v.double()
            w1 = w.double() - 1e-3 * m1
        assert all(close(got, placed(views(ref, 4))) for got, ref in zip(s, (w1, m1, v1)))
        one = [x.clone() for x in state[:3]]
        B.ws_shard_update(plan, -1, packed, *one, hy)
        mm, mv, master = state[1].clone(), state[2].clone(), w.clone()
        B.ws_fused_update(plan, -1, table, None, mm, mv, hy, B.TensorTable(plan, [views(master)]))
        assert all(torch.equal(a, b) for a, b in zip(one, s)) and torch.equal(mm, s[1]) and torch.equal(mv, s[2])
        back = torch.zeros_like(w)
        B.ws_unpack(plan, s[0], views(back))
        for o in outs + [master]:
            assert all(torch.equal(a, b) for a, b in zip(views(o), views(back)))
