"""Calls from several threads at once: a call on other objects or buffers
neither fails nor changes because another thread makes one of another size."""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2401_11324_gb300 as bang  # noqa: E402


def together(*calls):
    """Runs the calls in threads of their own, started together; raises what one raised."""
    gate, failed = threading.Barrier(len(calls)), []

    def run(call):
        gate.wait()
        try:
            call()
        except Exception as e:      # noqa: BLE001 -- handed to the test's thread
            failed.append(e)

    threads = [threading.Thread(target=run, args=(c,)) for c in calls]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    if failed:
        raise failed[0]


def test_table_layouts_of_several_sizes_at_once():
    # subspaces of one, two and four blocks of 16 dimensions need different
    # amounts of shared memory of the same kernel
    rng = np.random.default_rng(5)
    state = []
    for d, M in ((128, 32), (130, 32), (64, 1)):
        X = rng.integers(0, 256, size=(300, d)).astype(np.uint8)
        cb = (rng.normal(size=256 * d) * 60).astype(np.float32)
        h = bang.bang_create(0)
        bang.bang_load_pq(h, d, M, cb, np.zeros((300, M), np.uint8), 300)
        bang.bang_register_vectors(h, X, 0)
        q = torch.from_numpy(X[:130]).cuda()
        want = torch.empty((130, M, 256), device="cuda")
        bang.bang_pq_tables(h, q, 130, want)
        state.append((h, X, q, want, torch.empty_like(want), torch.cuda.Stream()))
    torch.cuda.synchronize()

    def call(s):
        h, _, q, want, out, stream = s
        for _ in range(1500):
            bang.bang_pq_tables(h, q, 130, out, 0, stream.cuda_stream)
        stream.synchronize()

    together(*[lambda s=s: call(s) for s in state])
    for h, _, _, want, out, _ in state:
        assert torch.equal(out, want)
        bang.bang_destroy(h)


@pytest.mark.parametrize("dt,ds", [("u8", (16, 128, 256)), ("f32", (16, 96, 208))])
def test_ground_truths_of_several_dimensions_at_once(dt, ds):
    state = []
    for d in ds:
        g = torch.Generator(device="cuda").manual_seed(d)
        X = torch.randint(0, 256, (70_000, d), generator=g, device="cuda")
        X = X.to({"u8": torch.uint8, "f32": torch.float32}[dt])
        q = X[:200].contiguous()
        state.append((X, q, bang.bang_ground_truth(X, q, 10)))

    def call(s):
        X, q, want = s
        stream = torch.cuda.Stream()
        for _ in range(30):
            ids, dist = bang.bang_ground_truth(X, q, 10, 0, stream.cuda_stream)
            assert (ids == want[0]).all() and (dist == want[1]).all()

    together(*[lambda s=s: call(s) for s in state])
