"""Child process of tests/test_gpu_bounds_checked.py: runs with BMU_LIBRARY pointing at the
bounds-checked build of the library (every id- and offset-derived address checked, violations
recorded in the status word instead of performed) and prints one JSON line."""
import ctypes
import json
import sys

import numpy as np
import torch

from inputs import synth
from tests import parity
from tests.test_gpu_screen import order_of, short_lists
import paper_2609_05138_b200 as bmu


def compare(*args):
    """parity.compare, with a failure turned into a count so that every case is reported"""
    try:
        return parity.compare(*args)
    except AssertionError as e:
        return {"docs": -1, "failed": 1, "detail": str(e)[:300]}


def status_word(ws):
    off = (-ws.data_ptr()) % 256
    return int(ws[off:off + 4].view(torch.int32)[0]) & 0xffffffff


def search(W, rp, ci, o, top2=False):
    D, M = W.shape
    N, nnz = rp.numel() - 1, ci.numel()
    need = max(bmu.bmu_search_workspace_bytes(D, M, N, nnz, o),
               int(bmu.load().bmu_search_top2_workspace_bytes(D, M, N, nnz, None)) * 2)
    ws = torch.zeros(need + 256, dtype=torch.uint8, device="cuda")
    if top2:
        out = bmu.bmu_search_top2_ws(W, rp, ci, opts=o, workspace=ws)
    else:
        out = bmu.bmu_search_ws(W, rp, ci, opts=o, workspace=ws)
    torch.cuda.synchronize()
    return out, status_word(ws)


def main():
    bmu.load()
    res = {"library": bmu.binding.load()._name, "clean": [], "flagged": []}
    cfg = synth.CONFIGS["cfg1"]
    rowptr, colidx = synth.make_corpus(cfg, n_docs=1500)
    rp, ci = rowptr.cuda(), colidx.cuda()
    for kernel, M, kw in ((1, 1000, {}), (3, 1024, {}), (4, 1024, {}), (6, 1024, {}),
                          (6, 1024 + 36, {"head_rows": 256, "chunk_neurons": 512, "relabel": 1}),
                          (6, 1024, {"tile_order": 2, "repack": 2})):
        W = synth.make_codebook(cfg.D, M, 40 + kernel, kind="scaled")
        o = bmu.Opts()
        o.kernel = kernel
        for k, v in kw.items():
            setattr(o, k, v)
        (ob, od), st = search(W.cuda(), rp, ci, o)
        r = compare(ob.cpu().numpy(), od.cpu().numpy(), W.numpy(), rowptr.numpy(), colidx.numpy())
        res["clean"].append({"kernel": kernel, "M": M, "status": st, "failed": r["failed"],
                             "docs": r["docs"], "detail": r.get("detail")})
    # second-best unit and the half-precision codebook through the tensor-core sweep
    W = synth.make_codebook(cfg.D, 1024, 7, kind="scaled")
    o = bmu.Opts()
    o.kernel = 6
    (b1, d1, b2, d2), st = search(W.cuda(), rp, ci, o, top2=True)
    r = compare(b1.cpu().numpy(), d1.cpu().numpy(), W.numpy(), rowptr.numpy(), colidx.numpy())
    res["clean"].append({"kernel": "6 top2", "M": 1024, "status": st, "failed": r["failed"], "docs": r["docs"]})
    W16 = W.cuda().half()
    ob, od = bmu.bmu_search_f16_ws(W16, rp, ci, opts=o)
    torch.cuda.synchronize()
    r = compare(ob.cpu().numpy(), od.cpu().numpy(), W16.float().cpu().numpy(), rowptr.numpy(),
                       colidx.numpy())
    res["clean"].append({"kernel": "6 f16", "M": 1024, "status": 0, "failed": r["failed"], "docs": r["docs"]})

    # the two-stage search: whole and ragged rows, a second-best unit, half precision, documents evaluated
    # whole (equal units, a long list), several launches; and the few-documents kernel
    few_rp, few_ci = rp[:301].contiguous(), ci[:int(rp[300])].contiguous()
    long_rp = torch.cat([rowptr, rowptr[-1:] + 1300])
    long_ci = torch.cat([colidx, torch.arange(0, 3 * 1300, 3, dtype=torch.int32)])
    res["two_stage"] = []
    for name, M, kind, kw in (("aligned", 1024, "scaled", {}), ("ragged", 1003, "scaled", {"chunk_neurons": 256}),
                              ("top2", 1028, "dupes", {"chunk_neurons": 256}), ("f16", 1024, "scaled", {}),
                              ("equal", 1003, "const", {}), ("long", 1024, "scaled", {"head_rows": 64}),
                              ("few", 1027, "scaled", {"two_stage": 0})):
        W = synth.make_codebook(cfg.D, M, 8, kind=kind).half().float()
        o = bmu.Opts()
        o.two_stage = 1
        for k, v in kw.items():
            setattr(o, k, v)
        r, c = (few_rp, few_ci) if name == "few" else (long_rp.cuda(), long_ci.cuda()) if name == "long" else (rp, ci)
        if name == "f16":
            need = int(bmu.load().bmu_search_f16_workspace_bytes(cfg.D, M, 1500, c.numel(), None))
            ws = torch.zeros(max(need, 1 << 26), dtype=torch.uint8, device="cuda")
            out = bmu.bmu_search_f16_ws(W.cuda().half(), r, c, opts=o, workspace=ws)
            torch.cuda.synchronize()
            st = status_word(ws)
        else:
            out, st = search(W.cuda(), r, c, o, top2=name == "top2")
        got = compare(out[0].cpu().numpy(), out[1].cpu().numpy(), W.numpy(), r.cpu().numpy(), c.cpu().numpy())
        res["two_stage"].append({"name": name, "status": st, "failed": got["failed"], "docs": got["docs"],
                                 "detail": got.get("detail")})
    # ... and with slabs in the order of the norms: whole and ragged rows, several launches, a second-best unit, half
    # precision; sets swept in the order of the map beside it, and documents evaluated whole
    res["by_norm"] = []
    for name, M, kw, every in (("aligned", 1024, {}, 50), ("ragged", 1027, {}, 0), ("top2", 1027, {}, 50),
                               ("launches", 3330, {"chunk_neurons": 640}, 0), ("f16", 1024, {}, 50)):
        r, c = (x.cuda() for x in short_lists(36_000, cfg.D, 9, every=every, extra=((300, 700),)))
        W = torch.rand((cfg.D, M), generator=torch.Generator().manual_seed(M)).half().float()
        norms = bmu.bmu_codebook_norms(W.cuda())
        o = bmu.Opts()
        o.two_stage = 1
        for k, v in kw.items():
            setattr(o, k, v)
        need = max(int(getattr(bmu.load(), "bmu_search_%sworkspace_bytes" % q)(cfg.D, M, 36_000, c.numel(), ctypes.byref(o)))
                   for q in ("top2_", "f16_"))
        ws = torch.zeros(need + 256, dtype=torch.uint8, device="cuda")
        if name == "f16":
            out = bmu.bmu_search_f16_ws(W.cuda().half(), r, c, norms=norms, opts=o, workspace=ws)
        else:
            call = bmu.bmu_search_top2_ws if name == "top2" else bmu.bmu_search_ws
            out = call(W.cuda(), r, c, norms=norms, opts=o, workspace=ws)
        torch.cuda.synchronize()
        got = compare(out[0].cpu().numpy(), out[1].cpu().numpy(), W.numpy(), r.cpu().numpy(), c.cpu().numpy())
        res["by_norm"].append({"name": name, "status": status_word(ws), "failed": got["failed"], "docs": got["docs"],
                               "detail": got.get("detail"), "order": order_of(ws, norms)})
    W = synth.make_codebook(cfg.D, 1024, 7, kind="scaled")

    # an id beyond the vocabulary: the checked build records it and leaves the access out.  The
    # codebook sits at the start of a larger allocation, so nothing here can leave memory that
    # the test owns.
    D, M = 3000, 1024
    big = torch.rand(D + 64, M, device="cuda")
    Wd = big[:D]
    bad = colidx.clone() % D
    bad[17] = D + 5
    for kernel in (1, 3, 4, 6):
        o = bmu.Opts()
        o.kernel = kernel
        _, st = search(Wd, rp, bad.cuda(), o)
        res["flagged"].append({"kernel": kernel, "status": st})
    for two_stage, (r, c) in ((1, (rp, bad.cuda())), (0, (few_rp, bad[:few_ci.numel()].cuda()))):
        o = bmu.Opts()
        o.two_stage = two_stage
        _, st = search(Wd, r, c, o)
        res["flagged"].append({"kernel": "two-stage" if two_stage else "few", "status": st})
    # the context is still usable and a clean search still passes
    o = bmu.Opts()
    o.kernel = 6
    (ob, od), st = search(W.cuda(), rp, ci, o)
    r = compare(ob.cpu().numpy(), od.cpu().numpy(), W.numpy(), rowptr.numpy(), colidx.numpy())
    res["after"] = {"status": st, "failed": r["failed"]}
    print(json.dumps(res))


if __name__ == "__main__":
    sys.exit(main())
