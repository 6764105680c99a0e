"""Calls on several streams, from several threads and in captured graphs at the same time: each has scratch of
its own, so the results are those of the calls alone."""
import threading

import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qnn():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1607_04683_gb300 import build, qnn as q
    build.build()
    q.lib()
    torch.cuda.set_device(0)
    return q


def matrix(rows, cols, seed):
    g = np.random.Generator(np.random.PCG64(seed))
    return (g.normal(0, 1, (rows, cols)) * (1 + seed)).astype(np.float32)


class Quantize:
    def __init__(self, qnn, rows, cols, seed):
        x = matrix(rows, cols, seed)
        self.qnn, self.x = qnn, torch.from_numpy(x).cuda()
        self.ref = [torch.from_numpy(np.ascontiguousarray(a).view(np.uint8)).cuda() for a in oracle.quantize(x, oracle.PER_MATRIX)]

    def run(self):
        return self.qnn.qnn_quantize(self.x, self.qnn.PER_MATRIX)

    def right(self, out):
        return all(torch.equal(a.reshape(-1).view(torch.uint8), b.reshape(-1)) for a, b in zip(out, self.ref))


class Product:
    """On the centered path (forced: the sizes are kept small for the oracle)."""

    def __init__(self, qnn, M, N, K, seed):
        ca, pa, ra = oracle.quantize(matrix(M, K, seed), oracle.PER_ROW)
        cw, pw, cs = oracle.quantize(matrix(N, K, seed + 1), oracle.PER_MATRIX)
        self.qnn = qnn
        self.args = (torch.from_numpy(ca).cuda(), qnn.params_tensor(pa), 1, torch.from_numpy(ra).cuda(),
                     torch.from_numpy(cw).cuda(), qnn.params_tensor(pw), torch.from_numpy(cs).cuda())
        self.ref = torch.from_numpy(oracle.qmatmul(ca, pa, 1, cw, pw)["y"]).cuda()

    def run(self):
        return self.qnn.qnn_qmatmul(*self.args)[0]

    def right(self, out):
        return torch.equal(out, self.ref)


@pytest.fixture()
def calls(qnn, monkeypatch):
    monkeypatch.setenv("QNN_QGEMM", "tc")
    c = [Quantize(qnn, 3000, 700, 1), Quantize(qnn, 20, 9000, 2), Quantize(qnn, 40000, 50, 3), Quantize(qnn, 3, 5, 4),
         Product(qnn, 300, 500, 600, 5), Product(qnn, 257, 130, 2100, 6), Product(qnn, 1000, 64, 100, 7)]
    torch.cuda.synchronize()
    return c


def test_streams(qnn, calls):
    streams = [torch.cuda.Stream() for _ in range(2 * len(calls))]
    outs = []
    for _ in range(12):
        for i, st in enumerate(streams):
            with torch.cuda.stream(st):
                outs.append((calls[i % len(calls)], calls[i % len(calls)].run()))
    torch.cuda.synchronize()
    assert all(c.right(o) for c, o in outs)
    assert qnn.device_status() == qnn.QNN_OK


def test_more_streams_than_slots(qnn, calls):
    streams = [torch.cuda.Stream(priority=p) for p in (0, -1, -2) for _ in range(32)]  # (torch has 32 of a priority)
    assert len({st.cuda_stream for st in streams}) > 64
    outs = []
    for st in streams:
        with torch.cuda.stream(st):
            for c in calls[:4]:
                outs.append((c, c.run()))
    torch.cuda.synchronize()
    assert all(c.right(o) for c, o in outs)


@pytest.mark.parametrize("shared", [False, True])
def test_threads(qnn, calls, shared):
    bad, one = [], torch.cuda.Stream()

    def work(i):
        st = one if shared else torch.cuda.Stream()
        with torch.cuda.stream(st):
            for k in range(30):
                c = calls[(i + k) % len(calls)]
                out = c.run()
                st.synchronize()
                if not c.right(out):
                    bad.append((i, k))

    threads = [threading.Thread(target=work, args=(i,)) for i in range(6)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad


def test_graphs_beside_eager_calls(qnn, calls):
    # captured without a call before them on their streams, replayed at the same time as one another and as eager calls
    graphs = []
    for c in calls:
        c.run()
    torch.cuda.synchronize()
    for c in calls + calls:
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            out = c.run()
        graphs.append((c, g, out, torch.cuda.Stream()))
    eager = []
    for _ in range(10):
        for i, (c, g, out, st) in enumerate(graphs):
            with torch.cuda.stream(st):
                g.replay()
        for c in calls:
            eager.append((c, c.run()))
    torch.cuda.synchronize()
    assert all(c.right(out) for c, _, out, _ in graphs)
    assert all(c.right(out) for c, out in eager)
