"""Every form of the search against the oracle, element by element.

The library chooses between one warp per query and a team of warps by the
queries that share an SM, so a test's small batch runs one of them only; here
the form is named, and the call says that it is the one that ran."""
import numpy as np
import pytest

import oracle
from tests import cases, forms

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2401_11324_gb300 as bang  # noqa: E402

# element types, dimensions on both sides of 128 and with and without 16-byte
# rows, uneven subspaces, rows on both sides of 64 neighbours
SETS = {
    "u8 128": dict(n=20_000, nq=300, ncomp=8),
    "u8 130": dict(n=5_000, nq=30, ncomp=4, dtype="u8", d=130, M=26, R=32, centre="uniform255"),
    "i8 100": dict(n=8_000, nq=40, ncomp=4, dtype="i8", d=100, M=30, R=40, centre="uniform100"),
    "i8 112": dict(n=5_000, nq=30, ncomp=4, dtype="i8", d=112, M=28, R=80, centre="uniform100"),
    "f32 96": dict(n=6_000, nq=50, ncomp=4, dtype="f32", d=96, M=48, R=68, centre="uniform255"),
    "f32 200": dict(n=5_000, nq=30, ncomp=4, dtype="f32", d=200, M=50, R=48, centre="uniform255"),
}
TRACE = 400


@pytest.fixture(scope="module", params=list(SETS))
def setup(request):
    w = cases.clustered(**SETS[request.param])
    ix = bang.Index(w["base"], w["codebook"], w["codes"], w["adj"], w["medoid"], w["M"])
    ref = oracle.Index(w["base"], w["codebook"], w["codes"], w["adj"], w["medoid"], w["M"])
    yield w, ix, ref
    ix.close()


def check(setup, mode, form, k, L, log2z=16, cap=0, placement=0, **kw):
    w, ix, ref = setup
    Q = np.ascontiguousarray(w["queries"][:40])
    nq = len(Q)
    ix.set_placement(placement)
    q = torch.from_numpy(Q).cuda()
    ids = torch.full((nq, k), -7, dtype=torch.int32, device="cuda")
    dist = torch.full((nq, k), -7.0, device="cuda")
    iters, status, ndist = (torch.full((nq,), -7, dtype=torch.int32, device="cuda") for _ in range(3))
    trace = torch.zeros((nq, TRACE), dtype=torch.int32, device="cuda")
    p = bang.make_params(mode=mode, bloom_log2=log2z, iter_cap=cap, out_iters=iters, out_status=status,
                         out_ndist=ndist, trace=trace, trace_cap=TRACE, **kw)
    ran = forms.search(ix, q, k, L, ids, dist, p, form=form)
    torch.cuda.synchronize()
    ix.set_placement(0)
    assert ran == form
    o = ref.search(Q, k, L, log2z=log2z, iter_cap=cap or None, trace_cap=TRACE, exact=mode == 2, q8=mode == 3,
                   bf16=mode == 1)
    assert (ids.cpu().numpy().view(np.uint32) == o["ids"]).all()
    fin = np.isfinite(o["dist"])
    got = dist.cpu().numpy()
    assert (np.isfinite(got) == fin).all() and (got[fin] == o["dist"][fin]).all()
    assert (iters.cpu().numpy() == o["iters"]).all() and (status.cpu().numpy() == o["status"]).all()
    assert (ndist.cpu().numpy().astype(np.uint64) == o["ndist"]).all()
    seen = np.arange(TRACE)[None] < np.minimum(o["iters"], TRACE)[:, None]
    assert (trace.cpu().numpy().view(np.uint32)[seen] == o["trace"][seen]).all()


@pytest.mark.parametrize("form", [1, 2, 3, 4])
@pytest.mark.parametrize("mode", [0, 1, 2, 3])
def test_form_equals_the_oracle(setup, mode, form):
    for k, L, log2z, cap in ((10, 48, 16, 0), (40, 90, 17, 0), (1, 3, 12, 0), (10, 40, 16, 9)):
        check(setup, mode, form, k, L, log2z, cap)


@pytest.mark.parametrize("form", [1, 3])
@pytest.mark.parametrize("mode", [0, 1, 2, 3])
@pytest.mark.parametrize("placement", [bang.BANG_NODE_RECORDS, bang.BANG_NODE_RECORDS | bang.BANG_GRAPH_PACKED,
                                       bang.BANG_GRAPH_IN_HBM | bang.BANG_VECTORS_IN_HBM | bang.BANG_GRAPH_PACKED])
def test_form_reads_every_placement(setup, mode, form, placement):
    check(setup, mode, form, 10, 48, placement=placement)


@pytest.mark.parametrize("mode", [0, 1, 2, 3])
@pytest.mark.parametrize("depth,early", [(2, 0), (0, 1), (2, 1)])
def test_one_warp_form_requests_ahead(setup, mode, depth, early):
    # the speculative request of the next entry and the early code rows, which
    # only this form has
    for placement in (0, bang.BANG_GRAPH_PACKED, bang.BANG_NODE_RECORDS):
        check(setup, mode, forms.ONE_WARP, 10, 64, placement=placement, prefetch_depth=depth, early_codes=early)
