"""Parity of the two-stage search (bmu_opts.two_stage = 1: an 8-bit image of the codebook screens
all units, what it cannot rule out is evaluated exactly in fp32) against the oracle, at the edges
of its tiles: documents per tile and block, units per group, slab and launch, heads that fill part
of a stage, lists that are empty, long, unsorted or repeat ids, and codebooks where nothing can be
ruled out."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
from inputs import synth
from tests import parity

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bmu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2609_05138_b200 as lib
    lib.load()
    return lib


def opts_of(bmu, **kw):
    o = bmu.Opts()
    o.two_stage = 1
    for k, v in kw.items():
        setattr(o, k, v)
    return o


def check(bmu, W, rowptr, colidx, floor=False, **kw):
    o = opts_of(bmu, **kw)
    Wd, rp, ci = W.cuda(), rowptr.cuda(), colidx.cuda()
    need = bmu.bmu_search_workspace_bytes(W.shape[0], W.shape[1], rp.numel() - 1, ci.numel(), o)
    ws = torch.zeros(need + 256, dtype=torch.uint8, device="cuda")
    ob, od = bmu.bmu_search_ws(Wd, rp, ci, opts=o, workspace=ws)
    torch.cuda.synchronize()
    off = (-ws.data_ptr()) % 256
    assert int(ws[off:off + 4].view(torch.int32)[0]) == 0                     # status word
    parity.compare(ob.cpu().numpy(), od.cpu().numpy(), W.numpy(), rowptr.numpy(), colidx.numpy(),
                   cancel_floor=floor)
    return ob, od


@pytest.mark.parametrize("n_docs", [1, 7, 8, 9, 127, 129])
@pytest.mark.parametrize("M", [1, 31, 33, 128, 300, 1003])
def test_edges_of_tiles_and_groups(bmu, n_docs, M):
    cfg = synth.CONFIGS["cfg1"]
    rowptr, colidx = synth.make_corpus(cfg, n_docs=n_docs)
    check(bmu, synth.make_codebook(cfg.D, M, 60, kind="scaled"), rowptr, colidx, chunk_neurons=256)


@pytest.mark.parametrize("D,head", [(1, 0), (63, 0), (65, 64), (300, 192), (4096, 64), (4096, 1536), (16384, 0),
                                    (16385, 0), (65024, 0)])
def test_edges_of_the_head(bmu, D, head):
    r = np.random.default_rng(D)
    rows = [r.permutation(D)[:int(r.integers(0, min(D, 60) + 1))] for _ in range(260)]
    rowptr = torch.zeros(len(rows) + 1, dtype=torch.int32)
    rowptr[1:] = torch.cumsum(torch.tensor([len(x) for x in rows]), 0)
    colidx = torch.from_numpy(np.concatenate(rows).astype(np.int32))
    check(bmu, synth.make_codebook(D, 700, 61, kind="signed"), rowptr, colidx, floor=True, head_rows=head)


@pytest.mark.parametrize("kind", ["uniform", "signed", "sparse", "dupes", "const", "prototype"])
def test_codebooks(bmu, kind):
    """dupes and const: exact ties, so the lowest index has to come through both stages."""
    cfg = synth.CONFIGS["cfg1"]
    rowptr, colidx = synth.make_corpus(cfg, n_docs=600)
    W = synth.make_codebook(cfg.D, 900, 62, kind=kind, docs=(rowptr, colidx))
    ob, _ = check(bmu, W, rowptr, colidx, floor=kind == "prototype", chunk_neurons=512)
    if kind == "dupes":
        assert int((ob % 2).sum()) == 0
    if kind == "const":
        assert int(ob.abs().sum()) == 0


def test_repeated_ids_and_lists_too_long_for_the_screen(bmu):
    """Repeated frequent ids stay out of the head; 300 ids lower the resolution of the image, and
    lists of more than 1040 gathered ids are evaluated whole."""
    D, M = 3000, 520
    r = np.random.default_rng(5)
    rows = [r.integers(0, D, 40), r.integers(0, 4, 30), r.permutation(D)[:1400], [], r.permutation(D)[:300]]
    rows = [np.asarray(x, dtype=np.int32) for x in rows] * 5
    rowptr = torch.zeros(len(rows) + 1, dtype=torch.int32)
    rowptr[1:] = torch.cumsum(torch.tensor([len(x) for x in rows]), 0)
    W = synth.make_codebook(D, M, 63, kind="scaled")
    for head in (64, 0):
        check(bmu, W, rowptr, torch.from_numpy(np.concatenate(rows)), head_rows=head)


def test_second_best_half_precision_and_plan(bmu):
    """The other entry points of the same two stages agree with the plain search and the oracle."""
    cfg = synth.CONFIGS["cfg3"]
    rowptr, colidx = synth.make_corpus(cfg, n_docs=700)
    g = torch.Generator().manual_seed(3)
    colidx = torch.randperm(cfg.D, generator=g).to(torch.int32)[colidx.long()]      # frequent ids anywhere
    W = synth.make_codebook(cfg.D, 1280, 64, kind="scaled").half().float()
    rp, ci, Wd, o = rowptr.cuda(), colidx.cuda(), W.cuda(), opts_of(bmu)
    ob, od = check(bmu, W, rowptr, colidx)
    b1, d1, b2, d2 = bmu.bmu_search_top2_ws(Wd, rp, ci, opts=o)
    assert torch.equal(b1, ob) and torch.equal(d1, od)
    e1, f1, e2, f2 = oracle.bmu2(W.numpy(), rowptr.numpy(), colidx.numpy())
    np.testing.assert_allclose(d2.cpu().numpy(), f2, rtol=1e-5)
    plan = bmu.Plan(rp, ci, cfg.D, 1280, o)
    pb, pd = plan.search(Wd)
    plan.close()
    assert torch.equal(pb, ob) and torch.equal(pd, od)
    hb, hd, hb2, hd2 = bmu.bmu_search_f16_ws(Wd.half(), rp, ci, opts=o, top2=True)
    assert torch.equal(hb, b1) and torch.equal(hd, d1) and torch.equal(hb2, b2) and torch.equal(hd2, d2)


@pytest.mark.parametrize("kind,M", [("const", 4096), ("dupes", 4096), ("ramp", 2304), ("steps", 4096)])
def test_lists_that_fill_over_many_launches(bmu, kind, M):
    """Launches of two slabs: a document's list fills up, is compacted when its minimum falls from
    launch to launch (ramp, steps), and overflows where nothing falls out of the window (const, dupes).
    Best and second-best unit and the half-precision codebook carry their minima between the launches."""
    cfg = synth.CONFIGS["cfg1"]
    rowptr, colidx = synth.make_corpus(cfg, n_docs=400)
    if kind in ("ramp", "steps"):
        # the same few features everywhere, a level that falls along the map
        level = torch.linspace(0.5, 0.0, M) if kind == "ramp" else torch.floor(torch.arange(M) / 512.0) * -0.03 + 0.5
        W = (0.2 * torch.rand((cfg.D, 1), generator=torch.Generator().manual_seed(9)) + level[None, :])
    else:
        W = synth.make_codebook(cfg.D, M, 67, kind=kind)
    W = W.half().float().contiguous()
    ob, od = check(bmu, W, rowptr, colidx, chunk_neurons=256)
    Wd, rp, ci, o = W.cuda(), rowptr.cuda(), colidx.cuda(), opts_of(bmu, chunk_neurons=256)
    args = (W.numpy(), rowptr.numpy(), colidx.numpy())
    b1, d1, b2, d2 = bmu.bmu_search_top2_ws(Wd, rp, ci, opts=o)
    parity.compare(b1.cpu().numpy(), d1.cpu().numpy(), *args)
    np.testing.assert_allclose(d2.cpu().numpy(), oracle.bmu2(*args)[3], rtol=1e-5)
    assert bool((b2 != b1).all())
    if kind == "const":                              # exact ties: the two lowest units
        assert int(b1.abs().max()) == 0 and int((b2 - 1).abs().max()) == 0
    h1, e1, h2, e2 = bmu.bmu_search_f16_ws(Wd.half(), rp, ci, opts=o, top2=True)
    parity.compare(h1.cpu().numpy(), e1.cpu().numpy(), *args)
    np.testing.assert_allclose(e2.cpu().numpy(), d2.cpu().numpy(), rtol=1e-6)


@pytest.mark.parametrize("M", [1, 40, 300, 1000, 1003, 2304])
@pytest.mark.parametrize("f16", [False, True])
def test_documents_evaluated_whole(bmu, M, f16):
    """Every unit within the window of every document (equal units), lists that end in every place of a batch
    of 64 ids or 8 rows: best and second-best unit, whole and ragged rows and slabs."""
    if f16 and M % 256:
        pytest.skip("half precision takes whole slabs of 256 units")
    D = 2000
    r = np.random.default_rng(12)
    rows = [np.sort(r.permutation(D)[:n]) for n in (0, 1, 7, 8, 9, 63, 64, 65, 71, 72, 128, 200, 1100)] * 3
    rowptr = torch.zeros(len(rows) + 1, dtype=torch.int32)
    rowptr[1:] = torch.cumsum(torch.tensor([len(x) for x in rows]), 0)
    colidx = torch.from_numpy(np.concatenate(rows).astype(np.int32))
    W = torch.rand((D, 1), generator=torch.Generator().manual_seed(2)).expand(D, M)
    W = (W * (1 + 1e-3 * (torch.arange(M) // 100 % 2))[None, :]).half().float().contiguous()
    Wd, rp, ci, o = W.cuda(), rowptr.cuda(), colidx.cuda(), opts_of(bmu, chunk_neurons=512)
    args = (W.numpy(), rowptr.numpy(), colidx.numpy())
    if f16:
        b1, d1, b2, d2 = bmu.bmu_search_f16_ws(Wd.half(), rp, ci, opts=o, top2=True)
    else:
        check(bmu, W, rowptr, colidx, chunk_neurons=512)
        b1, d1, b2, d2 = bmu.bmu_search_top2_ws(Wd, rp, ci, opts=o)
    parity.compare(b1.cpu().numpy(), d1.cpu().numpy(), *args)
    if M == 1:
        assert int(b2.max()) == -1 and bool(torch.isinf(d2).all())
    else:
        e2 = oracle.bmu2(*args)[3]
        np.testing.assert_allclose(d2.cpu().numpy(), e2, rtol=1e-5)
        assert bool((b2 != b1).all())


@pytest.mark.parametrize("how", ["weights", "norms"])
def test_distances_that_are_not_finite(bmu, how):
    """A unit at infinity is never chosen; where all are, the answer is the single-stage kernels' one."""
    cfg = synth.CONFIGS["cfg1"]
    rowptr, colidx = synth.make_corpus(cfg, n_docs=200)
    W = synth.make_codebook(cfg.D, 768, 69, kind="scaled")
    far = list(range(0, 768, 3))
    if how == "weights":
        W[5, far] = 3e38                              # its norm and the row's range overflow
    Wd, rp, ci = W.cuda(), rowptr.cuda(), colidx.cuda()
    norms = bmu.bmu_codebook_norms(Wd)
    if how == "norms":
        norms[far] = float("inf")
    assert bool(torch.isinf(norms[far]).all()) and int(torch.isinf(norms).sum()) == len(far)
    single = bmu.Opts()
    single.kernel, single.two_stage = 3, 2
    for n in (norms, torch.full_like(norms, float("inf"))):
        ob, od = bmu.bmu_search_ws(Wd, rp, ci, norms=n, opts=opts_of(bmu))
        rb, rd = bmu.bmu_search_ws(Wd, rp, ci, norms=n, opts=single)
        assert torch.equal(ob, rb)
        assert torch.equal(torch.isinf(od), torch.isinf(rd))
        ok = ~torch.isinf(rd)
        assert bool(((od - rd).abs() <= 1e-5 * rd.abs())[ok].all())


def timed(bmu, W, rp, ci, two_stage, norms=None):
    o = bmu.Opts()
    o.two_stage = two_stage
    need = bmu.bmu_search_workspace_bytes(W.shape[0], W.shape[1], rp.numel() - 1, ci.numel(), o)
    ws = torch.empty(need + 256, dtype=torch.uint8, device="cuda")
    ms = []
    for _ in range(8):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        bmu.bmu_search_ws(W, rp, ci, opts=o, workspace=ws, norms=norms)
        b.record()
        torch.cuda.synchronize()
        ms.append(a.elapsed_time(b))
    return min(ms[2:])


@pytest.mark.parametrize("what,most", [("equal units", 2.8), ("an outlier", 2.8), ("long lists", 1.5),
                                       ("some long lists", 0.8)])
def test_where_the_screen_cannot_rule_out_it_costs_little(bmu, what, most):
    """The automatic choice against the single-stage one, where nothing (or for some documents nothing) can
    be ruled out: at most the screening and, once more, all units.  Evaluated by scattered groups instead of
    whole it was 5.4, 8.0, 3.0 and 2.9 times as long."""
    D, M, dev = 16384, 4096, torch.device("cuda")
    g = torch.Generator(device=dev).manual_seed(6)
    n = 60_000 if what == "some long lists" else 20_000
    lens = torch.full((n,), 80, dtype=torch.int64, device=dev)
    if what == "long lists":
        n, lens = 5_000, lens[:5_000] * 25
    rp, ci = synth.draw_corpus(n, D, 1.1 if what != "long lists" else 0.2, lens, 6, dev)
    if what == "some long lists":
        extra = torch.cat([torch.randperm(D, generator=g, device=dev)[:3000].sort().values for _ in range(60)])
        rp = torch.cat([rp, rp[-1] + 3000 * torch.arange(1, 61, dtype=torch.int32, device=dev)])
        ci = torch.cat([ci, extra.to(torch.int32)])
    if what == "equal units":
        W = torch.rand((D, 1), generator=g, device=dev).expand(D, M).contiguous()
    else:
        W = synth.make_codebook(D, M, 3, dev)
    if what == "an outlier":
        W[D - 5, 77] = 1000.0
    assert bmu.bmu_describe_search(D, M, rp.numel() - 1, ci.numel()).two_stage
    assert timed(bmu, W, rp, ci, 0) <= most * timed(bmu, W, rp, ci, 2)


def test_units_at_infinity_do_not_widen_the_windows(bmu):
    """Norms that rule units out (masked units, weights whose square overflows): screened like any other map,
    where every document used to be evaluated whole (1.6 times the single-stage search; 0.5 without them)."""
    D, M, dev = 16384, 4096, torch.device("cuda")
    rp, ci = synth.draw_corpus(20_000, D, 1.1, torch.full((20_000,), 80, dtype=torch.int64, device=dev), 6, dev)
    W = synth.make_codebook(D, M, 3, dev)
    norms = bmu.bmu_codebook_norms(W)
    norms[::5] = float("inf")
    ob, od = bmu.bmu_search_ws(W, rp, ci, norms=norms)
    keep = [j for j in range(M) if j % 5]
    rb, rd = bmu.bmu_search_ws(W[:, keep].contiguous(), rp, ci)
    assert torch.equal(ob, torch.tensor(keep, dtype=torch.int32, device=dev)[rb.long()])
    assert bool(((od - rd).abs() <= 1e-5 * rd.abs()).all())
    assert timed(bmu, W, rp, ci, 0, norms) <= 0.9 * timed(bmu, W, rp, ci, 2, norms)


def smooth_map(bmu, rp, ci, D, edge):
    """A map after one update from random units with the widest neighbourhood."""
    M, dev = edge * edge, rp.device
    unit = torch.randint(0, M, (rp.numel() - 1,), generator=torch.Generator(device=dev).manual_seed(3), device=dev,
                         dtype=torch.int32)
    num = torch.zeros((D, M), dtype=torch.int32, device=dev)
    cnt = torch.zeros(M, dtype=torch.int32, device=dev)
    W = torch.zeros((D, M), device=dev)
    bmu.bmu_update_scatter(rp, ci, unit, num, cnt)
    bmu.bmu_update_writeback(*bmu.bmu_update_blur(num, cnt, edge, edge, 8.0), W)
    return W


@pytest.mark.parametrize("f16", [False, True])
def test_nothing_is_screened_where_most_documents_are_evaluated_whole(bmu, f16):
    """Equal units on 128 x 128: little more than the single-stage search.  A smooth map whose units lie close
    together: same units up to near ties; the plan, the batches of a call and half precision take the same way."""
    D, edge, dev = 16384, 128, torch.device("cuda")
    rp, ci = synth.draw_corpus(20_000, D, 1.1, torch.full((20_000,), 80, dtype=torch.int64, device=dev), 6, dev)
    W = smooth_map(bmu, rp, ci, D, edge)
    if f16:
        Wh = W.half()
        hb, hd = bmu.bmu_search_f16_ws(Wh, rp, ci)
        ob, od = bmu.bmu_search_ws(Wh.float(), rp, ci)
        assert torch.equal(hb, ob) and torch.equal(hd, od)
        return
    ob, od = bmu.bmu_search_ws(W, rp, ci)
    some = list(range(0, 20_000, 400))
    parity.compare(ob.cpu().numpy(), od.cpu().numpy(), W.cpu().numpy(), rp.cpu().numpy(), ci.cpu().numpy(), docs=some)
    plan = bmu.Plan(rp, ci, D, edge * edge)
    pb, pd = plan.search(W)
    plan.close()
    assert torch.equal(pb, ob) and torch.equal(pd, od)
    host = (rp.cpu().pin_memory(), ci.cpu().pin_memory())
    for hb, hd in bmu.bmu_search_batches_host(W, [host, host]):
        assert torch.equal(hb, ob.cpu()) and torch.equal(hd, od.cpu())
    W.copy_(W[:, :1].clone().expand(D, edge * edge))
    assert timed(bmu, W, rp, ci, 0) <= 1.9 * timed(bmu, W, rp, ci, 2)


def test_a_long_list_costs_the_others_nothing(bmu):
    """One list of 1000 ids among ordinary ones: neither the codes of all others nor the time of their tiles
    follow it (1.67 -> 3.05 ms when they did); what is left is the walk along the one list.  Same results, the
    long one among them."""
    D, M, n, dev = 16384, 16384, 20_000, torch.device("cuda")
    g = torch.Generator(device=dev).manual_seed(6)
    rp, ci = synth.draw_corpus(n, D, 1.1, torch.full((n,), 80, dtype=torch.int64, device=dev), 6, dev)
    more = torch.randperm(D, generator=g, device=dev)[:1000].sort().values.to(torch.int32)
    rpl, cil = torch.cat([rp, rp[-1:] + 1000]), torch.cat([ci, more])
    W = synth.make_codebook(D, M, 3, dev)
    o = opts_of(bmu)
    ob, od = bmu.bmu_search_ws(W, rp, ci, opts=o)
    lb, ld = bmu.bmu_search_ws(W, rpl, cil, opts=o)
    assert torch.equal(lb[:n], ob) and torch.equal(ld[:n], od)
    parity.compare(lb.cpu().numpy(), ld.cpu().numpy(), W.cpu().numpy(), rpl.cpu().numpy(), cil.cpu().numpy(),
                   docs=[0, 1, n])
    more, without = timed(bmu, W, rpl, cil, 1), timed(bmu, W, rp, ci, 1)
    assert more <= without + 0.9, (more, without)


@pytest.mark.parametrize("n,fewer", [(45_500, 45_000), (45_500, 9_000), (2_500, 1_500), (2_500, 300)])
def test_a_workspace_for_more_documents_serves_fewer(bmu, n, fewer):
    """Best unit, second-best unit and half precision with the workspace of a larger search."""
    cfg = synth.CONFIGS["cfg1"]
    W = synth.make_codebook(cfg.D, 1024, 68, kind="scaled").half().float().cuda()
    lens = synth.draw_nnz("poisson", 80.0, n, torch.Generator().manual_seed(4), "cpu")
    rp, ci = (x.cuda() for x in synth.draw_corpus(n, cfg.D, 1.0, lens, 4, "cpu"))
    small = (rp[:fewer + 1].contiguous(), ci[:int(rp[fewer])].contiguous())
    lib = bmu.load()
    for query, search, Wd in (("", bmu.bmu_search_ws, W), ("top2_", bmu.bmu_search_top2_ws, W),
                              ("f16_", bmu.bmu_search_f16_ws, W.half())):
        need = int(getattr(lib, "bmu_search_%sworkspace_bytes" % query)(cfg.D, 1024, n, ci.numel(), None))
        ws = torch.empty(need + 256, dtype=torch.uint8, device="cuda")
        got = [x.clone() for x in search(Wd, *small, workspace=ws)]
        own = search(Wd, *small)
        assert all(torch.equal(a, b) for a, b in zip(got, own))


def test_batches_share_the_images_of_the_codebook(bmu):
    """Batches of one call: the second has lists that the images of the first are too fine for, the
    third lists other features, the fourth takes another route.  Every result as by itself."""
    D, M = 3000, 2048
    r = np.random.default_rng(8)
    perm = r.permutation(D)

    def corpus(n, skew, long_lists=0, names=None):
        rows = [np.unique((D * r.random(70) ** skew).astype(np.int32)) for _ in range(n)]
        for i in range(long_lists):
            rows[7 * i] = np.sort(r.permutation(np.arange(D // 2, D))[:900]).astype(np.int32)
        if names is not None:
            rows = [names[x].astype(np.int32) for x in rows]
        rp = np.concatenate([[0], np.cumsum([len(x) for x in rows])]).astype(np.int32)
        return torch.from_numpy(rp).pin_memory(), torch.from_numpy(np.concatenate(rows)).pin_memory()

    batches = [corpus(7000, 2.5), corpus(7300, 2.5, long_lists=40), corpus(7001, 2.5, names=perm),
               corpus(300, 2.5), corpus(7100, 2.5)]
    W = synth.make_codebook(D, M, 66, kind="scaled").cuda()
    outs = bmu.bmu_search_batches_host(W, batches)
    assert bmu.bmu_last_status() == (0, 0)
    for (rp, ci), (ob, od) in zip(batches, outs):
        assert rp.numel() < 1000 or bmu.bmu_describe_search(D, M, rp.numel() - 1, ci.numel()).two_stage
        rb, rd = bmu.bmu_search(W, rp.cuda(), ci.cuda())
        assert torch.equal(rb.cpu(), ob) and torch.equal(rd.cpu(), od)


@pytest.mark.parametrize("n,more", [(1, 0), (4000, 0), (60_000, 4)])
def test_nothing_is_launched_for_an_order_that_cannot_pay(bmu, n, more):
    """A map of 1,024 units, from which on norms are looked at, against one of 1,023: the order kernel, the images, the
    sweep and the verification of slabs by norm only where the whole sweep takes longer than these cost."""
    D, dev = 4096, torch.device("cuda")
    rp, ci = synth.draw_corpus(n, D, 1.0, torch.full((n,), 64, dtype=torch.int64, device=dev), 3, dev)
    launches = []
    for M in (1023, 1024):
        W = torch.rand((D, M), generator=torch.Generator(device=dev).manual_seed(4), device=dev)
        norms = bmu.bmu_codebook_norms(W)
        before = bmu.bmu_kernel_launches()
        bmu.bmu_search_ws(W, rp, ci, norms=norms, opts=opts_of(bmu))
        launches.append(bmu.bmu_kernel_launches() - before)
    assert launches[1] - launches[0] == more, launches


def test_a_large_codebook_shares_its_images(bmu):
    """640,000 units of 1,536 features: 1.97 GB of images in the order of the map, which batches share, and as many as
    a quarter of them again in the order of the norms, which must not keep the former from being shared."""
    D, M, n, dev = 1536, 640_000, 1100, torch.device("cuda")
    rp, ci = synth.draw_corpus(n, D, 1.0, torch.full((n,), 80, dtype=torch.int64, device=dev), 3, dev)
    W = torch.rand((D, M), generator=torch.Generator(device=dev).manual_seed(4), device=dev)
    assert bmu.bmu_describe_search(D, M, n, ci.numel()).two_stage
    batch = (rp.cpu().pin_memory(), ci.cpu().pin_memory())

    def launches(call):
        before = bmu.bmu_kernel_launches()
        out = call()
        return bmu.bmu_kernel_launches() - before, out

    norms, _ = launches(lambda: bmu.bmu_codebook_norms(W))
    one, (first,) = launches(lambda: bmu.bmu_search_batches_host(W, [batch]))
    two, both = launches(lambda: bmu.bmu_search_batches_host(W, [batch, batch]))
    assert two < 2 * one - norms                     # no ranges and no choice of the head for the second batch
    for ob, od in both:
        assert torch.equal(ob, first[0]) and torch.equal(od, first[1])
    bmu.bmu_release_scratch()


def lists(lens, D, seed):
    r = np.random.default_rng(seed)
    rows = [np.sort(r.permutation(D)[:n]) for n in lens]
    rowptr = torch.zeros(len(rows) + 1, dtype=torch.int32)
    rowptr[1:] = torch.cumsum(torch.tensor([len(x) for x in rows]), 0)
    return rowptr, torch.from_numpy(np.concatenate(rows).astype(np.int32))


@pytest.mark.parametrize("M,chunk", [(1024, 0), (1027, 256), (2304, 1024), (5000, 512)])
@pytest.mark.parametrize("n_docs", [1, 129, 700])
def test_slabs_in_the_order_of_the_norms(bmu, M, chunk, n_docs):
    """Norms that spread further than a document reaches: short lists on an iid U[0,1) codebook.  Some lists are
    empty, some reach half of the map, one all of it; best and second-best unit, half precision, a plan.  So few that
    the order of the norms cannot pay and none is made: the same lists by the thousand further down."""
    D = 4096
    r = np.random.default_rng(M + n_docs)
    lens = r.integers(0, 24, n_docs)
    lens[::50] = 60
    if n_docs > 300:
        lens[300] = 900
    rowptr, colidx = lists(lens, D, M)
    W = torch.rand((D, M), generator=torch.Generator().manual_seed(M)).half().float()
    ob, od = check(bmu, W, rowptr, colidx, chunk_neurons=chunk)
    Wd, rp, ci, o = W.cuda(), rowptr.cuda(), colidx.cuda(), opts_of(bmu, chunk_neurons=chunk)
    b1, d1, b2, d2 = bmu.bmu_search_top2_ws(Wd, rp, ci, opts=o)
    assert torch.equal(b1, ob)
    np.testing.assert_allclose(d2.cpu().numpy(), oracle.bmu2(W.numpy(), rowptr.numpy(), colidx.numpy())[3], rtol=1e-6)
    assert bool((b2 != b1).all())
    plan = bmu.Plan(rp, ci, D, M, o) if M % 4 == 0 else None
    if plan:
        pb, pd = plan.search(Wd)
        plan.close()
        assert torch.equal(pb, ob) and torch.equal(pd, od)
    if M % 256 == 0:
        hb, hd = bmu.bmu_search_f16_ws(Wd.half(), rp, ci, opts=o)[:2]
        assert torch.equal(hb, ob) and torch.equal(hd, od)


@pytest.mark.parametrize("copies", [2, 40, 1500])
def test_equal_units_in_the_order_of_the_norms(bmu, copies):
    """The unit of the smallest norm many times over the map: the lowest index wins, the next one is second (300
    documents: in the order of the map; where norms are in order, further down)."""
    D, M = 4096, 4096
    rowptr, colidx = lists(np.random.default_rng(3).integers(0, 24, 300), D, 4)
    W = torch.rand((D, M), generator=torch.Generator().manual_seed(5))
    W[:, 7] = 0.98 * W[:, int((W ** 2).sum(0).argmin())]
    where = 7 + (4000 // copies) * torch.arange(copies)
    W[:, where] = W[:, 7:8]
    check(bmu, W, rowptr, colidx)
    b1, d1, b2, d2 = bmu.bmu_search_top2_ws(W.cuda(), rowptr.cuda(), colidx.cuda(), opts=opts_of(bmu))
    assert bool((b1 == 7).all()) and bool((b2 == int(where[1])).all())
    assert torch.equal(d1, d2)


@pytest.mark.parametrize("value", [float("inf"), float("-inf"), float("nan")])
def test_norms_that_have_no_place_in_an_order(bmu, value):
    """A unit at plus infinity or without a number as its norm never wins; at minus infinity it always does (200
    documents: in the order of the map; where norms are in order, further down)."""
    D, M = 4096, 2048
    rowptr, colidx = lists(np.random.default_rng(6).integers(1, 24, 200), D, 7)
    W = torch.rand((D, M), generator=torch.Generator().manual_seed(8))
    Wd, rp, ci = W.cuda(), rowptr.cuda(), colidx.cuda()
    norms = bmu.bmu_codebook_norms(Wd)
    far = int(norms.argmin())
    norms[far] = value
    ob, od = bmu.bmu_search_ws(Wd, rp, ci, norms=norms, opts=opts_of(bmu))
    if value < 0:
        assert bool((ob == far).all()) and bool(torch.isinf(od).all())
    else:
        keep = [j for j in range(M) if j != far]
        rb, rd = bmu.bmu_search_ws(Wd[:, keep].contiguous(), rp, ci, opts=opts_of(bmu))
        assert torch.equal(ob, rb + (rb >= far).int())
        assert bool(((od - rd).abs() <= 1e-5 * rd.abs()).all())


def test_batches_that_reach_further_than_the_first(bmu):
    """Batches share order and images: one whose lists reach further than the first one's, one of long lists only,
    which needs the slabs in the order of the map, and a short one again (a few thousand documents; so many that
    slabs are in the order of the norms, further down)."""
    D, M = 4096, 4096
    W = torch.rand((D, M), generator=torch.Generator().manual_seed(9)).cuda()
    r = np.random.default_rng(10)
    batches = [lists(lens, D, 11 + i) for i, lens in enumerate((r.integers(0, 16, 3000), r.integers(10, 50, 3000),
                                                                 r.integers(200, 500, 2000), r.integers(0, 16, 3000)))]
    outs = [(torch.empty(rp.numel() - 1, dtype=torch.int32).pin_memory(),
             torch.empty(rp.numel() - 1, dtype=torch.float32).pin_memory()) for rp, _ in batches]
    bmu.bmu_search_batches_host(W, [(rp.pin_memory(), ci.pin_memory()) for rp, ci in batches], outs)
    single = bmu.Opts()
    single.two_stage = 2
    for (rp, ci), (ob, od) in zip(batches, outs):
        rb, rd = bmu.bmu_search_ws(W, rp.cuda(), ci.cuda(), opts=single)
        parity.compare(ob.numpy(), od.numpy(), W.cpu().numpy(), rp.numpy(), ci.numpy(), docs=np.arange(0, 2000, 97))
        assert float((ob == rb.cpu()).float().mean()) > 0.999
        assert bool(((od - rd.cpu()).abs() <= 1e-5 * rd.cpu().abs()).all())


def added_as_documented(W, norms, rowptr, colidx, whole_rows):
    """Distances with a unit's weights in partial sums over every 16th id (32nd: fp16; 4th: rows that are not whole
    16-byte pieces), added in pairs, all in fp32.  (The 64-bit sum under a rounding to 32 is the fused one.)"""
    parts = 4 if not whole_rows else 32 if W.dtype == np.float16 else 16
    bmu, dist = [], []
    for i in range(len(rowptr) - 1):
        ids = colidx[rowptr[i]:rowptr[i + 1]]
        s = np.zeros((parts, W.shape[1]), dtype=np.float32)
        for e, f in enumerate(ids):
            s[e % parts] += W[f].astype(np.float32)
        while len(s) > 1:
            s = s[:len(s) // 2] + s[len(s) // 2:] if whole_rows else s[0::2] + s[1::2]
        d = (norms.astype(np.float64) - 2.0 * s[0].astype(np.float64)).astype(np.float32)
        bmu.append(int(d.argmin()))
        dist.append(np.float32(len(ids)) + d.min())
    return np.array(bmu, dtype=np.int32), np.array(dist, dtype=np.float32)


@pytest.mark.parametrize("M,f16", [(1280, False), (1003, False), (1280, True)])
def test_a_distance_is_the_same_whichever_way_it_was_evaluated(bmu, M, f16):
    """The same documents by themselves, where candidates are verified, and among twice as many long lists, where
    all documents are evaluated whole: the same bits, and those of the order of additions that is documented."""
    D = 3000
    r = np.random.default_rng(21)
    lens = [0, 1, 3, 4, 5, 7, 15, 16, 17, 31, 32, 33, 47, 48, 63, 64, 65, 80, 81, 127, 128, 129, 200, 300]
    some, many = lists(lens, D, 22), lists(lens + [int(n) for n in r.integers(1100, 1400, 2 * len(lens) + 8)], D, 22)
    W = torch.rand((D, M), generator=torch.Generator().manual_seed(23)) * torch.rand((D, 1), generator=torch.Generator().manual_seed(24))
    W = W.cuda().half() if f16 else W.cuda()
    norms = (bmu.bmu_codebook_norms_f16 if f16 else bmu.bmu_codebook_norms)(W)
    search = bmu.bmu_search_f16_ws if f16 else bmu.bmu_search_ws
    n = len(lens)
    want = added_as_documented(W.cpu().numpy(), norms.cpu().numpy(), some[0].numpy(), some[1].numpy(), M % 4 == 0)
    for rowptr, colidx in (some, many):
        assert torch.equal(colidx[:some[1].numel()], some[1])
        ob, od = search(W, rowptr.cuda(), colidx.cuda(), norms=norms, opts=opts_of(bmu, head_rows=64))[:2]
        np.testing.assert_array_equal(ob[:n].cpu().numpy(), want[0])
        np.testing.assert_array_equal(od[:n].cpu().numpy(), want[1])


def test_a_document_is_answered_alike_in_any_company(bmu):
    """Documents on both sides of the reach up to which slabs are swept in the order of the norms: the whole corpus,
    parts of it (which draw the line elsewhere), other chunks, a plan, and the same call again."""
    D, M, n, dev = 16384, 4096, 120_000, torch.device("cuda")
    lens = synth.draw_nnz("poisson", 80.0, n, torch.Generator(device=dev).manual_seed(4), dev)
    rp, ci = synth.draw_corpus(n, D, 1.0, lens, 4, dev)
    W = synth.make_codebook(D, M, 5, dev)
    ob, od = bmu.bmu_search_ws(W, rp, ci)
    same = [bmu.bmu_search_ws(W, rp, ci) for _ in range(3)]
    same += [bmu.bmu_search_ws(W, rp, ci, opts=opts_of(bmu, chunk_neurons=c)) for c in (512, 1024)]
    plan = bmu.Plan(rp, ci, D, M)
    same.append(plan.search(W))
    parts = [bmu.bmu_search_ws(W, (rp[a:b + 1] - rp[a]).contiguous(), ci[int(rp[a]):int(rp[b])].contiguous(), opts=opts_of(bmu))
             for a, b in ((0, 30_000), (30_000, 37_000), (37_000, n))]
    same.append([torch.cat([x[i] for x in parts]) for i in (0, 1)])
    for k, (sb, sd) in enumerate(same):
        assert torch.equal(sb, ob) and torch.equal(sd, od), (k, int((sb != ob).sum()), int((sd != od).sum()))
    plan.close()


# ---- ... with so many documents that slabs are in the order of the norms ----------------------------
def order_of(ws, norms):
    """What a search decided, from its workspace: None where its slabs followed the map, else (units in the order of the
    norms, sets of documents swept in the order of the map beside it, documents evaluated whole).  Found by what stands in
    front of it: the units of the smallest norm at even and at odd indices, and four words on those norms."""
    off = (-ws.data_ptr()) % 256
    words = ws[off:off + (ws.numel() - off) // 4 * 4].view(torch.int32)
    floats = words.view(torch.float32)
    finite = torch.where(torch.isfinite(norms), norms, torch.full_like(norms, float("inf")))
    even, odd = 2 * int(finite[0::2].argmin()), 2 * int(finite[1::2].argmin()) + 1
    found = (words[:-8] == even) & (words[1:-7] == odd) & (floats[4:-4] == norms[even]) & (floats[5:-3] == norms[odd])
    (at,) = found.nonzero().flatten().tolist()
    base = at - 16
    return (int(words[base + 19]), int(words[base + 22]), int(words[38])) if int(words[base + 12]) else None


def scratch(query, *sizes):
    return torch.zeros(int(query(*sizes)) + 256, dtype=torch.uint8, device="cuda")


def short_lists(n, D, seed, every=50, length=60, extra=()):
    """n lists of 0 .. 23 ids, every 50th of 60 ids, and some given ones: CPU tensors."""
    g = torch.Generator().manual_seed(seed)
    lens = torch.randint(0, 24, (n,), generator=g)
    if every:
        lens[::every] = length
    for at, m in extra:
        lens[at] = m
    return drawn(lens, D, seed)


def drawn(lens, D, seed, s=0.05):
    rowptr, colidx = synth.draw_corpus(lens.numel(), D, s, lens, seed, "cuda")
    return rowptr.cpu(), colidx.cpu()


@pytest.mark.parametrize("M,chunk,n,few_far", [(1024, 0, 40_000, False), (1027, 0, 40_000, False), (2304, 1024, 30_000, True),
                                               (5000, 512, 12_000, False), (3331, 640, 24_000, True)])
def test_many_documents_in_the_order_of_the_norms(bmu, M, chunk, n, few_far):
    """Whole and ragged rows, last slabs that are not full, one launch and several; lists that reach far by the
    hundred, whose sets are swept in the order of the map (or a handful, which are evaluated whole), one that
    reaches all of the map and one that no sum holds.  Best and second-best unit, half precision, a plan."""
    D = 4096
    rowptr, colidx = short_lists(n, D, M, every=0 if few_far else 50, extra=((300, 700), (301, 1300)))
    W = torch.rand((D, M), generator=torch.Generator().manual_seed(M)).half().float()
    Wd, rp, ci, o = W.cuda(), rowptr.cuda(), colidx.cuda(), opts_of(bmu, chunk_neurons=chunk)
    norms = bmu.bmu_codebook_norms(Wd)
    args = (W.numpy(), rowptr.numpy(), colidx.numpy())
    lib, by = bmu.load(), ctypes.byref(o)
    ws = scratch(lib.bmu_search_workspace_bytes, D, M, n, ci.numel(), by)
    ob, od = bmu.bmu_search_ws(Wd, rp, ci, norms=norms, opts=o, workspace=ws)
    parity.compare(ob.cpu().numpy(), od.cpu().numpy(), *args)
    kept, by_map, whole = order_of(ws, norms)
    assert 0 < kept < M and (whole > 0 if few_far else by_map > 0), (kept, by_map, whole)
    again = bmu.bmu_search_ws(Wd, rp, ci, norms=norms, opts=o, workspace=ws)
    assert torch.equal(again[0], ob) and torch.equal(again[1], od)
    ws = scratch(lib.bmu_search_top2_workspace_bytes, D, M, n, ci.numel(), by)
    b1, d1, b2, d2 = bmu.bmu_search_top2_ws(Wd, rp, ci, norms=norms, opts=o, workspace=ws)
    assert order_of(ws, norms)
    assert torch.equal(b1, ob) and torch.equal(d1, od) and bool((b2 != b1).all())
    np.testing.assert_allclose(d2.cpu().numpy(), oracle.bmu2(*args)[3], rtol=1e-6)
    if M % 4 == 0:
        plan = bmu.Plan(rp, ci, D, M, o)
        pb, pd = plan.search(Wd, norms=norms)
        assert order_of(plan.workspace, norms)
        plan.close()
        assert torch.equal(pb, ob) and torch.equal(pd, od)
    if M % 256 == 0:
        ws = scratch(lib.bmu_search_f16_workspace_bytes, D, M, n, ci.numel(), by)
        hb, hd = bmu.bmu_search_f16_ws(Wd.half(), rp, ci, norms=norms, opts=o, workspace=ws)[:2]
        assert order_of(ws, norms)
        parity.compare(hb.cpu().numpy(), hd.cpu().numpy(), *args)


@pytest.mark.parametrize("copies,step,ordered", [(2, 0.0, True), (40, 0.0, True), (200, 0.0, True), (700, 5e-8, True), (700, 0.0, False)])
def test_equal_and_nearly_equal_units_by_norm(bmu, copies, step, ordered):
    """Neighbours of the smallest norm: the lowest index wins, the next one is second.  700 units of nearly that norm lie
    in the windows of all but the shortest lists, in 22 places where a document's list holds 16; 700 equal norms have no
    order that sorting by counting finds, and the slabs follow the map."""
    D, M, n = 4096, 8192, 12_000
    rowptr, colidx = short_lists(n, D, 4, every=0)
    W = torch.rand((D, M), generator=torch.Generator().manual_seed(5))
    W[:, 7] = 0.98 * W[:, int((W ** 2).sum(0).argmin())]
    where = 7 + torch.arange(copies)
    W[:, where] = W[:, 7:8] * (1 + step * torch.arange(copies)[None, :])
    Wd, rp, ci, o = W.cuda(), rowptr.cuda(), colidx.cuda(), opts_of(bmu)
    norms = bmu.bmu_codebook_norms(Wd)
    lib, by = bmu.load(), ctypes.byref(o)
    ws = scratch(lib.bmu_search_workspace_bytes, D, M, n, ci.numel(), by)
    ob, od = bmu.bmu_search_ws(Wd, rp, ci, norms=norms, opts=o, workspace=ws)
    args = (W.numpy(), rowptr.numpy(), colidx.numpy())
    parity.compare(ob.cpu().numpy(), od.cpu().numpy(), *args)
    got = order_of(ws, norms)
    assert bool(got) == ordered
    if copies == 700 and ordered:
        assert got[2] > n // 3                       # evaluated whole: their lists were too short
    ws = scratch(lib.bmu_search_top2_workspace_bytes, D, M, n, ci.numel(), by)
    b1, d1, b2, d2 = bmu.bmu_search_top2_ws(Wd, rp, ci, norms=norms, opts=o, workspace=ws)
    assert bool(order_of(ws, norms)) == ordered
    assert torch.equal(b1, ob) and torch.equal(d1, od) and bool((b2 != b1).all())
    np.testing.assert_allclose(d2.cpu().numpy(), oracle.bmu2(*args)[3], rtol=1e-6)
    if not step:
        assert bool((b1 == 7).all()) and bool((b2 == 8).all()) and torch.equal(d1, d2)


@pytest.mark.parametrize("value,ordered", [(float("inf"), True), (float("nan"), True), (float("-inf"), False)])
def test_many_documents_and_norms_that_have_no_place(bmu, value, ordered):
    """Some units at plus infinity or without a number as their norm never win, and the others are in order; one at
    minus infinity always wins, and the slabs follow the map."""
    D, M, n = 4096, 2050, 24_000
    rowptr, colidx = short_lists(n, D, 7, every=0)
    W = torch.rand((D, M), generator=torch.Generator().manual_seed(8))
    Wd, rp, ci, o = W.cuda(), rowptr.cuda(), colidx.cuda(), opts_of(bmu)
    norms = bmu.bmu_codebook_norms(Wd)
    far = norms.argsort()[:1 if value < 0 else 5].sort().values
    norms[far] = value
    ws = scratch(bmu.load().bmu_search_workspace_bytes, D, M, n, ci.numel(), ctypes.byref(o))
    ob, od = bmu.bmu_search_ws(Wd, rp, ci, norms=norms, opts=o, workspace=ws)
    if value < 0:
        assert bool((ob == far[0]).all()) and bool(torch.isinf(od).all())
        return
    assert bool(order_of(ws, norms)) == ordered
    keep = torch.ones(M, dtype=torch.bool, device="cuda")
    keep[far] = False
    left = keep.nonzero().flatten()
    rb, rd = bmu.bmu_search_ws(Wd[:, left].contiguous(), rp, ci, norms=norms[left].contiguous(), opts=o)
    assert torch.equal(ob, left[rb.long()].int())
    assert bool(((od - rd).abs() <= 1e-6 * rd.abs()).all())


def test_many_batches_that_reach_further_than_the_first(bmu):
    """Batches share order and images: lists that reach further than the first one's, long lists only, which need the
    slabs in the order of the map, short ones again (order and images stand), and some that lower the steps of
    the image, so that both images are made anew."""
    D, M = 16384, 4096
    W = torch.rand((D, M), generator=torch.Generator().manual_seed(9)).cuda()
    norms = bmu.bmu_codebook_norms(W)
    g = torch.Generator().manual_seed(10)
    batches = []
    for k, (n, lo, hi) in enumerate(((24_000, 20, 36), (20_000, 30, 60), (6_000, 300, 500), (24_500, 20, 36), (24_000, 20, 36), (23_000, 20, 40))):
        lens = torch.randint(lo, hi, (n,), generator=g)
        if k == 4:
            lens[::100] = 800
        batches.append(drawn(lens, D, 11 + k))
    ordered, want = [], []
    for rp, ci in batches:
        assert bmu.bmu_describe_search(D, M, rp.numel() - 1, ci.numel()).two_stage
        ws = scratch(bmu.load().bmu_search_workspace_bytes, D, M, rp.numel() - 1, ci.numel(), None)
        want.append(bmu.bmu_search_ws(W, rp.cuda(), ci.cuda(), norms=norms, workspace=ws))
        ordered.append(bool(order_of(ws, norms)))
    assert ordered == [True, True, False, True, True, True]
    outs = bmu.bmu_search_batches_host(W, [(rp.pin_memory(), ci.pin_memory()) for rp, ci in batches])
    for (rp, ci), (ob, od), (rb, rd) in zip(batches, outs, want):
        assert torch.equal(ob, rb.cpu()) and torch.equal(od, rd.cpu())
        parity.compare(ob.numpy(), od.numpy(), W.cpu().numpy(), rp.numpy(), ci.numpy(), docs=np.arange(0, rp.numel() - 1, 97))


@pytest.mark.parametrize("kind", ["by norm", "by map", "whole"])
def test_captured_in_a_graph(bmu, kind):
    """Launches that begin under the end of the one before stay in order when they are captured and replayed, in either
    order of slabs and with documents evaluated whole, on other weights in the same buffers."""
    D, M, n = 4096, 2304, 24_000
    rowptr, colidx = short_lists(n, D, 14, every=0) if kind == "by norm" else \
        drawn(torch.full((n,), 64, dtype=torch.int64), D, 14, 1.0)
    rp, ci, o = rowptr.cuda(), colidx.cuda(), opts_of(bmu, chunk_neurons=1024)
    W = synth.make_codebook(D, M, 73, kind="const" if kind == "whole" else "uniform").cuda()
    other = synth.make_codebook(D, M, 74, kind="uniform").cuda()
    ws = scratch(bmu.load().bmu_search_workspace_bytes, D, M, n, ci.numel(), ctypes.byref(o))
    want = [bmu.bmu_search_ws(x, rp, ci, opts=o, workspace=ws) for x in (W, other)]
    assert bool(order_of(ws, bmu.bmu_codebook_norms(other))) == (kind == "by norm")
    buf, ob, od = W.clone(), torch.empty(n, dtype=torch.int32, device="cuda"), torch.empty(n, device="cuda")
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        bmu.bmu_search_ws(buf, rp, ci, opts=o, workspace=ws, out_bmu=ob, out_dist=od)
    for x, (wb, wd) in ((W, want[0]), (other, want[1]), (W, want[0])):
        buf.copy_(x)
        ob.fill_(-1)
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(ob, wb) and torch.equal(od, wd)
