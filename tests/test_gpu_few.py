"""Parity of the few-documents kernel (the automatic choice below about a thousand documents: no
tiling pass, the neuron axis spread over the grid, a ticket per document) against the oracle, at the
edges of its slabs and pieces, aligned and ragged, best and second-best unit, one-shot and planned."""
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


@pytest.mark.parametrize("n_docs,M", [(1, 1), (1, 3), (3, 127), (4, 128), (5, 129), (48, 252), (48, 256),
                                      (300, 260), (300, 2048), (1000, 1025), (1000, 4100)])
def test_few_documents_match_the_oracle(bmu, n_docs, M):
    cfg = synth.CONFIGS["cfg5"]                        # lists of 1 .. 400 ids
    rowptr, colidx = synth.make_corpus(cfg, n_docs=n_docs)
    W = synth.make_codebook(cfg.D, M, 70, kind="scaled")
    Wd, rp, ci = W.cuda(), rowptr.cuda(), colidx.cuda()
    n0 = bmu.bmu_kernel_launches()
    ob, od = bmu.bmu_search(Wd, rp, ci)
    assert bmu.bmu_kernel_launches() - n0 == 2         # norms and the search
    torch.cuda.synchronize()
    args = (W.numpy(), rowptr.numpy(), colidx.numpy())
    parity.compare(ob.cpu().numpy(), od.cpu().numpy(), *args)
    b1, d1, b2, d2 = bmu.bmu_search_top2_ws(Wd, rp, ci)
    assert torch.equal(b1, ob) and torch.equal(d1, od)
    if M == 1:
        assert int(b2.max()) == -1 and bool(torch.isinf(d2).all())
    else:
        np.testing.assert_allclose(d2.cpu().numpy(), oracle.bmu2(*args)[3], rtol=1e-5)
    plan = bmu.Plan(rp, ci, cfg.D, M)
    pb, pd = plan.search(Wd)
    plan.close()
    assert torch.equal(pb, ob) and torch.equal(pd, od)


def test_empty_repeated_and_unaligned(bmu):
    """Empty rows, repeated and unsorted ids, a codebook that starts off a 16-byte boundary."""
    r = np.random.default_rng(1)
    D, M = 900, 512
    rows = [[], r.permutation(D)[:31], r.integers(0, D, 33), r.permutation(D)[:700], r.integers(0, 3, 9)] * 7
    rowptr = torch.zeros(len(rows) + 1, dtype=torch.int32)
    rowptr[1:] = torch.cumsum(torch.tensor([len(x) for x in rows]), 0)
    colidx = torch.from_numpy(np.concatenate(rows).astype(np.int32))
    W = synth.make_codebook(D, M, 71, kind="signed")
    buf = torch.empty(D * M + 1, device="cuda")
    off = buf[1:].view(D, M)
    off.copy_(W)
    for Wd in (W.cuda(), off):
        ob, od = bmu.bmu_search_ws(Wd, rowptr.cuda(), colidx.cuda())
        torch.cuda.synchronize()
        parity.compare(ob.cpu().numpy(), od.cpu().numpy(), W.numpy(), rowptr.numpy(), colidx.numpy(),
                       cancel_floor=True)


@pytest.mark.parametrize("n_docs,M", [(48, 512), (700, 65_536)])
def test_one_shot_reads_back_where_it_pays_and_can_be_captured(bmu, n_docs, M):
    """The one-shot search agrees with the workspace form, whether it knows the number of listings (large
    maps) or not, and is still captured in a graph."""
    r = np.random.default_rng(3)
    D = 400
    rows = [np.sort(r.permutation(D)[:int(r.integers(1, 60))]) for _ in range(n_docs)]
    rp = torch.zeros(n_docs + 1, dtype=torch.int32)
    rp[1:] = torch.cumsum(torch.tensor([len(x) for x in rows]), 0)
    rp, ci = rp.cuda(), torch.from_numpy(np.concatenate(rows).astype(np.int32)).cuda()
    W = synth.make_codebook(D, M, 72, kind="scaled").cuda()
    ob, od = bmu.bmu_search(W, rp, ci)
    wb, wd = bmu.bmu_search_ws(W, rp, ci)
    assert torch.equal(ob, wb) and torch.equal(od, wd)
    graph = torch.cuda.CUDAGraph()
    gb, gd = torch.empty_like(ob), torch.empty_like(od)
    with torch.cuda.graph(graph):
        bmu.bmu_search(W, rp, ci, gb, gd)
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(gb, ob) and torch.equal(gd, od)
