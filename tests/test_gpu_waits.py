"""The team form's bounded waits: when one gives up (a query's first expander
answers nothing, and waits may last half a millisecond instead of seconds), that query
reports it, the queries that follow in the same CTA are searched as ever, and
callers that read no status of each query return an error."""
import numpy as np
import pytest

from tests import cases, forms

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2401_11324_gb300 as bang  # noqa: E402

SHORT = 1_000_000               # SM cycles: far above any expansion, far below the batches


@pytest.fixture(scope="module")
def u8small():
    return cases.clustered(n=20_000, nq=300, ncomp=8)


@pytest.mark.parametrize("mode,log2z", [(0, 16), (3, 16), (2, 17)])
@pytest.mark.parametrize("expanders", [1, 2, 3])
def test_a_wait_that_gives_up_ends_its_query_only(u8small, mode, log2z, expanders):
    w = u8small
    nq, silent = 30_000, 7      # many queries for each CTA of the persistent launch
    Q = np.resize(w["queries"], (nq, 128))
    ix = bang.Index(w["base"], w["codebook"], w["codes"], w["adj"], w["medoid"], w["M"])
    q = torch.from_numpy(np.ascontiguousarray(Q)).cuda()
    kq = torch.full((nq,), 10, dtype=torch.int32, device="cuda")
    Lq = torch.full((nq,), 64, dtype=torch.int32, device="cuda")
    got = []
    for mute, wait in ((None, 0), (silent, SHORT)):
        out = dict(ids=torch.full((nq, 10), -7, dtype=torch.int32, device="cuda"),
                   dist=torch.full((nq, 10), -7.0, device="cuda"),
                   iters=torch.zeros(nq, dtype=torch.int32, device="cuda"),
                   status=torch.full((nq,), 9, dtype=torch.int32, device="cuda"))
        p = bang.make_params(mode=mode, bloom_log2=log2z, out_iters=out["iters"], out_status=out["status"])
        ran = forms.search(ix, q, 10, 64, out["ids"], out["dist"], p, kq, Lq, 1 + expanders, wait, mute)
        torch.cuda.synchronize()
        assert ran == 1 + expanders
        got.append({k: v.cpu().numpy() for k, v in out.items()})
    ix.close()
    ref, cut = got
    assert (ref["status"] == 0).all()
    assert cut["status"][silent] == 3 and (np.delete(cut["status"], silent) == 0).all()
    for f in ("ids", "dist", "iters"):
        assert (np.delete(cut[f], silent, 0) == np.delete(ref[f], silent, 0)).all(), f


def test_server_reports_a_wait_that_gave_up(u8small):
    w = u8small
    ix = bang.Index(w["base"], w["codebook"], w["codes"], w["adj"], w["medoid"], w["M"])
    k, L = np.full(50, 10, np.uint32), np.full(50, 64, np.uint32)
    want = np.zeros((50, 10), np.uint32), np.zeros((50, 10), np.float32)
    ix.search_batched(w["queries"][:50], k, L, 10, 64, *want)
    srv = bang.Server(ix, 10, 64, max_batch=64, streams=2)
    try:
        for mute in (None, 3, None):
            forms.server_form(srv, 3, SHORT if mute is not None else 0, mute)
            t = srv.submit(w["queries"][:50], k, L)
            if mute is None:
                ids, dist, _ = srv.wait(t, 20_000)
                assert (ids == want[0]).all() and (dist == want[1]).all()
            else:
                with pytest.raises(bang.BangError, match="gave up") as e:
                    srv.wait(t, 20_000)
                assert e.value.code == bang.BANG_ECUDA
    finally:
        srv.stop()
        ix.close()


def test_graph_build_reports_a_wait_that_gave_up(u8small):
    X = u8small["base"][:3000]
    centres = X[::1000].astype(np.float32)
    want, _ = bang.bang_build_shard_graph(X, centres, 2, 32, 32, 1.2, 0.05, 14)
    with pytest.raises(bang.BangError, match="gave up") as e:
        forms.shard_graph(X, centres, 2, 32, 32, 1.2, 0.05, 14, 3, SHORT, 0)
    assert e.value.code == bang.BANG_ETIMEOUT
    assert (forms.shard_graph(X, centres, 2, 32, 32, 1.2, 0.05, 14, 3) == want).all()
