"""The persistent tensor-core stack (lstm_persist.cu) against the oracle, bit for bit: every layer's
outputs, final states and 8-bit logits, at the edges of its tiles (rows of a quarter, of one and two row
tiles), of a block's cells (odd and even numbers of cells, cells past the last block) and of its
reductions, rows outside the fp32 form, carried states, host buffers, streams and repeated calls."""
import numpy as np
import pytest

import oracle
import parity

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


@pytest.fixture(autouse=True)
def persist(monkeypatch):
    monkeypatch.setenv("QNN_LSTM_PATH", "persist")


def workload(L=2, I=40, H=64, C=0, B=5, T=4, mode=1, w=0.2):
    from paper_1607_04683_gb300 import inputs
    return inputs.LstmWorkload("persist", seed=L + H + B, num_layers=L, input_dim=I, hidden=H, proj=0, num_classes=C,
                               batch=B, frames=T, w_range=w, forget_bias=1.0, seq_mean_range=0.5,
                               output_mode=mode if C else 0, out_w_range=0.5)


def model_of(qnn, wl, params):
    d = qnn.lstm_desc(wl.num_layers, wl.input_dim, wl.hidden, 0, wl.num_classes, wl.output_mode)
    return qnn.LstmModel(d, torch.from_numpy(params).cuda())


def reference(wl, params, x, **kw):
    d = oracle.desc(wl.num_layers, wl.input_dim, wl.hidden, 0, wl.num_classes, wl.output_mode)
    return oracle.lstm_forward(d, params, x, want_h_all=True, want_logits=wl.num_classes > 0, **kw)


def forward(qnn, model, wl, x, h=None, c=None, h_all=True):
    B, T, _ = x.shape
    L, H, C = wl.num_layers, wl.hidden, wl.num_classes
    dev = dict(dtype=torch.float32, device="cuda")
    hs = torch.from_numpy(h).cuda() if h is not None else torch.zeros((L, B, H), **dev)
    cs = torch.from_numpy(c).cuda() if c is not None else torch.zeros((L, B, H), **dev)
    ha = torch.full((L, B, T, H), float("nan"), **dev) if h_all else None
    lg = torch.full((B, T, C), float("nan"), **dev) if C else None
    y = model.forward(torch.from_numpy(np.ascontiguousarray(x)).cuda(), h_state=hs, c_state=cs, h_all=ha, logits=lg)
    assert qnn.device_status() == qnn.QNN_OK
    out = {"y": y.cpu().numpy(), "h": hs.cpu().numpy(), "c": cs.cpu().numpy()}
    if h_all:
        out["h_all"] = ha.cpu().numpy()
    if lg is not None:
        out["logits"] = lg.cpu().numpy()
    return out


def check(qnn, wl, got, ref, params):
    w_out = wl.out_weights(params) if wl.num_classes else None
    parity.compare(got, ref, wl.num_layers, wl.num_classes, wl.output_mode, w_out)
    if wl.num_classes == 0:
        assert np.array_equal(got["y"], ref["h_all"][-1])


CASES = [dict(L=1, I=1, H=1, B=1, T=3), dict(L=1, I=8, H=8, B=5, T=3), dict(L=2, H=7, B=8, C=5), dict(L=2, H=100, B=17, C=9),
         dict(L=3, H=128, B=32, C=50), dict(L=2, H=300, B=33), dict(L=2, H=301, B=64, C=20), dict(L=5, H=500, B=16, T=6, C=200, w=0.08),
         dict(L=4, H=512, B=65, T=3, w=0.08), dict(L=2, H=128, B=128, C=20), dict(L=2, H=129, B=129), dict(L=3, I=320, H=450, B=200, T=3, w=0.08),
         dict(L=5, H=500, B=256, T=3, C=20, w=0.08), dict(L=1, I=600, H=1000, B=9, T=3, w=0.05), dict(L=8, H=64, B=40, T=5),
         dict(L=2, H=64, B=9, C=10, mode=2),
         # the plan's other forms: 16, 20 and 24 cells a block with one, two and four quarters in use
         dict(L=4, H=512, B=30, T=2, w=0.08), dict(L=4, H=510, B=50, T=2, w=0.08), dict(L=5, H=498, B=60, T=2, w=0.08),
         dict(L=5, H=500, B=100, T=2, w=0.08), dict(L=8, H=384, B=20, T=2, C=30, w=0.1), dict(L=8, H=383, B=40, T=2, w=0.1),
         dict(L=8, H=384, B=100, T=2, w=0.1)]


@pytest.mark.parametrize("cfg", CASES)
def test_stack_bit_exact(qnn, cfg):
    wl = workload(**cfg)
    params, x = wl.make()
    ref = reference(wl, params, x)
    qnn.profile_read()
    qnn.profile_enable(True)
    model = model_of(qnn, wl, params)
    got = forward(qnn, model, wl, x)
    qnn.profile_enable(False)
    assert "lstm_persist" in qnn.profile_read()
    check(qnn, wl, got, ref, params)
    # without the layer outputs, and carried states: two calls in a row equal one
    plain = forward(qnn, model, wl, x, h_all=False)
    assert np.array_equal(plain["y"], got["y"]) and np.array_equal(plain["h"], got["h"])
    a = forward(qnn, model, wl, x[:, :1], h_all=False)
    b = forward(qnn, model, wl, x[:, 1:], h=a["h"], c=a["c"], h_all=False)
    assert np.array_equal(b["h"], got["h"]) and np.array_equal(b["c"], got["c"])
    assert np.array_equal(np.concatenate([a["y"], b["y"]], 1), got["y"])


# Two row tiles of blocks of 24 cells have no tensor memory: such a stack stays on the layer wavefront.
@pytest.mark.parametrize("H,B", [(384, 130), (384, 256), (381, 129)])
def test_stack_without_a_plan(qnn, H, B, monkeypatch):
    monkeypatch.delenv("QNN_LSTM_PATH")
    wl = workload(L=8, H=H, B=B, T=2, w=0.1)
    params, x = wl.make()
    model = model_of(qnn, wl, params)
    qnn.profile_read()
    qnn.profile_enable(True)
    got = forward(qnn, model, wl, x)
    qnn.profile_enable(False)
    assert "lstm_persist" not in qnn.profile_read()
    b = [0, 63, 127, 128, B - 1]
    ref = reference(wl, params, np.ascontiguousarray(x[b]))
    assert np.array_equal(got["h_all"][:, b], ref["h_all"]) and np.array_equal(got["c"][:, b], ref["c"])


@pytest.mark.parametrize("B", [9, 150])
@pytest.mark.parametrize("offset,scale", [(50.0, 0.01), (-3000.0, 1.0), (1.0e6, 1.0)])
def test_rows_outside_the_fp32_form(qnn, B, offset, scale):
    # inputs far from zero for their spread: large offsets z, sums that need 64 bits, units without a range
    wl = workload(L=2, H=64, B=B, C=10)
    params, x = wl.make()
    x[::2] = (x[::2] * scale + offset).astype(np.float32)
    check(qnn, wl, forward(qnn, model_of(qnn, wl, params), wl, x), reference(wl, params, x), params)


def test_saturated_gates(qnn):
    # pre-activations beyond the short exponential's range
    wl = workload(L=2, H=40, B=33, w=40.0)
    params, x = wl.make()
    check(qnn, wl, forward(qnn, model_of(qnn, wl, params), wl, x), reference(wl, params, x), params)


def test_repeated_calls_of_other_sizes(qnn):
    wl = workload(L=2, H=96, B=70, T=9, C=12)
    params, x = wl.make()
    model = model_of(qnn, wl, params)
    ref = reference(wl, params, x)
    for B, T in ((70, 9), (3, 2), (33, 9), (70, 1), (70, 9)):
        got = forward(qnn, model, wl, x[:B, :T])
        assert np.array_equal(got["h_all"], ref["h_all"][:, :B, :T])
        assert np.array_equal(got["logits"], ref["logits"][:B, :T])


def test_host_buffers(qnn):
    wl = workload(L=2, H=48, B=20, T=5, C=300)
    params, x = wl.make()
    model = model_of(qnn, wl, params)
    dev = forward(qnn, model, wl, x, h_all=False)
    assert np.array_equal(model.forward(x), dev["y"])
    y = torch.full((20, 5, 300), float("nan")).pin_memory()
    lg = torch.full((20, 5, 300), float("nan")).pin_memory()
    h, c = np.zeros((2, 20, 48), np.float32), np.zeros((2, 20, 48), np.float32)
    ha = np.zeros((2, 20, 5, 48), np.float32)
    model.forward(torch.from_numpy(x).pin_memory(), y=y, h_state=h, c_state=c, h_all=ha, logits=lg)
    torch.cuda.synchronize()
    assert np.array_equal(y.numpy(), dev["y"]) and np.array_equal(lg.numpy(), dev["logits"])
    assert np.array_equal(h, dev["h"]) and np.array_equal(c, dev["c"])
    assert np.array_equal(ha, reference(wl, params, x)["h_all"])


def test_two_models_on_two_streams(qnn):
    # launches of two models overlap in time only as far as both grids fit: results are theirs alone
    pairs = []
    for H, B in ((300, 40), (500, 100)):
        wl = workload(L=3, H=H, B=B, T=20, w=0.08)
        params, x = wl.make()
        pairs.append((model_of(qnn, wl, params), torch.from_numpy(x).cuda(), torch.cuda.Stream()))
    alone = [m.forward(x).clone() for m, x, _ in pairs]
    torch.cuda.synchronize()
    outs = [[], []]
    for _ in range(5):
        for i, (m, x, st) in enumerate(pairs):
            with torch.cuda.stream(st):
                outs[i].append(m.forward(x))
    torch.cuda.synchronize()
    assert qnn.device_status() == qnn.QNN_OK
    for i in range(2):
        for y in outs[i]:
            assert torch.equal(y, alone[i])


def test_non_finite_input_is_reported(qnn):
    wl = workload(L=2, H=64, B=20, C=5)
    params, x = wl.make()
    model = model_of(qnn, wl, params)
    bad = x.copy()
    bad[3, 1, 2] = np.nan
    model.forward(torch.from_numpy(bad).cuda())
    assert qnn.device_status() == qnn.QNN_ERR_NONFINITE
    check(qnn, wl, forward(qnn, model, wl, x), reference(wl, params, x), params)


def test_replayed_graph(qnn):
    wl = workload(L=2, H=96, B=24, T=6, C=12)
    params, x = wl.make()
    model = model_of(qnn, wl, params)
    xg = torch.from_numpy(x).cuda()
    y = torch.empty((24, 6, 12), device="cuda")
    model.forward(xg, y=y)  # weights and workspace are made before the capture
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        model.forward(xg, y=y, stream=torch.cuda.current_stream())
    for k in range(3):
        xk = np.roll(x, k, 0)
        xg.copy_(torch.from_numpy(xk))
        y.fill_(float("nan"))
        g.replay()
        torch.cuda.synchronize()
        parity.check_posteriors(y.cpu().numpy(), reference(wl, params, xk)["y"])


# Where the persistent stack cannot run, automatic dispatch hands the call to the path that took it before.
def test_refused_cooperative_launch(qnn, monkeypatch):
    monkeypatch.delenv("QNN_LSTM_PATH")
    monkeypatch.setenv("QNN_NO_COOP", "1")
    wl = workload(L=2, H=64, B=70, C=12)
    params, x = wl.make()
    model = model_of(qnn, wl, params)
    qnn.profile_read()
    qnn.profile_enable(True)
    got = forward(qnn, model, wl, x)
    qnn.profile_enable(False)
    assert "lstm_gates_tc" in qnn.profile_read()
    check(qnn, wl, got, reference(wl, params, x), params)
    with pytest.raises(qnn.QnnError) as e:  # the layerwise kernel's launch is cooperative too
        model.forward(torch.from_numpy(x[:20]).cuda())
    assert e.value.status == qnn.QNN_ERR_NO_COOP
    monkeypatch.delenv("QNN_NO_COOP")
    check(qnn, wl, forward(qnn, model, wl, x), reference(wl, params, x), params)


def least_memory(qnn, monkeypatch, run):
    """The least QNN_MODEL_MEMORY (to 1%) with which run() succeeds."""
    lo, hi = 0, 1 << 28
    while hi - lo > hi // 100:
        mid = (lo + hi) // 2
        monkeypatch.setenv("QNN_MODEL_MEMORY", str(mid))
        try:
            run()
            hi = mid
        except qnn.QnnError as e:
            assert e.status == qnn.QNN_ERR_NO_MEMORY
            lo = mid
    monkeypatch.delenv("QNN_MODEL_MEMORY")
    return hi


def test_posteriors_that_fit_only_chunk_by_chunk(qnn, monkeypatch):
    monkeypatch.setenv("QNN_OUT_CHUNK", "1")
    wl = workload(L=2, H=64, B=130, T=8, C=2000)
    params, x = wl.make()
    xd = torch.from_numpy(x).cuda()
    y = torch.empty((130, 8, 2000)).pin_memory()

    def run(path):
        monkeypatch.setenv("QNN_LSTM_PATH", path)
        model_of(qnn, wl, params).forward(xd, y=y)
        torch.cuda.synchronize()

    least = {path: least_memory(qnn, monkeypatch, lambda: run(path)) for path in ("tc", "persist")}
    assert 1.2 * least["tc"] < least["persist"]
    run("persist")
    ref = y.clone()
    monkeypatch.setenv("QNN_MODEL_MEMORY", str((least["tc"] + least["persist"]) // 2))
    y.fill_(float("nan"))
    run("auto")
    assert torch.equal(y, ref)  # (both sum a row's terms in one order)


def test_memory_of_the_persistent_stack_is_given_back(qnn, monkeypatch):
    monkeypatch.delenv("QNN_LSTM_PATH")
    wl = workload(L=2, H=128, B=300, T=8)
    params, x = wl.make()
    xd = torch.from_numpy(x).cuda()
    ref = model_of(qnn, wl, params).forward(xd)
    least = least_memory(qnn, monkeypatch, lambda: model_of(qnn, wl, params).forward(xd))
    model = model_of(qnn, wl, params)
    monkeypatch.setenv("QNN_MODEL_MEMORY", str(least))
    small = model.forward(xd[:100])  # the persistent stack
    assert torch.equal(model.forward(xd), ref)  # the wavefront, whose buffers fit only without it
    assert torch.equal(model.forward(xd[:100]), small)  # (on whichever has room)


# Logits leave in one pass over them, whatever the frames, into any kind of buffer and at any alignment.
@pytest.mark.parametrize("where", ["device", "pinned", "pageable"])
@pytest.mark.parametrize("B,T,C,off", [(1, 1, 1, 0), (5, 40, 7, 1), (20, 3, 300, 0), (40, 9, 12, 1), (130, 2, 64, 0)])
def test_logits_in_sequence_order(qnn, B, T, C, off, where):
    wl = workload(L=1 if B < 5 else 2, H=24, B=B, T=T, C=C)
    params, x = wl.make()
    buf = torch.full((off + B * T * C + 1,), 7.0, device="cuda" if where == "device" else "cpu")
    buf = buf.pin_memory() if where == "pinned" else buf
    lg = buf[off:-1].reshape(B, T, C)
    model = model_of(qnn, wl, params)
    xd, y = torch.from_numpy(x).cuda(), torch.empty((B, T, C), device="cuda")
    qnn.profile_read()
    qnn.profile_enable(True)
    model.forward(xd, y=y, logits=lg)
    torch.cuda.synchronize()
    qnn.profile_enable(False)
    assert qnn.profile_read()["rows_to_sequences"][0] == 1
    assert np.array_equal(lg.cpu().numpy(), reference(wl, params, x)["logits"])
    assert float(buf[-1]) == 7.0 and (off == 0 or float(buf[0]) == 7.0)
