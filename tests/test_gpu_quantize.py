"""The quantizer kernels at the edges of their splits, against the oracle: rows around the register
kernel's widths and its rows per wave, matrices around the range pass's segments and the code pass's
long rows, unaligned and strided inputs, rows after others in one warp."""
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


def check(qnn, x, ld, off, granularity, static=False):
    rows, cols = x.shape
    buf = torch.full((off + rows * ld,), float("nan"), device="cuda")
    v = buf[off:].reshape(rows, ld)[:, :cols]
    v.copy_(torch.from_numpy(x))
    if static:
        codes, params, sums = (torch.empty(n, dtype=t, device="cuda") for n, t in (((rows, cols), torch.uint8), ((1, 4), torch.int32),
                                                                                   (rows, torch.int32)))
        assert qnn.lib().qnn_quantize_matrix_static(v.data_ptr(), rows, cols, ld, codes.data_ptr(), cols, params.data_ptr(),
                                                    sums.data_ptr(), None, None) == qnn.QNN_OK
    else:
        codes, params, sums = qnn.qnn_quantize(v, granularity)
    assert qnn.device_status() == qnn.QNN_OK
    c, p, s = oracle.quantize(x, granularity)
    assert np.array_equal(codes.cpu().numpy(), c)
    assert np.array_equal(qnn.params_view(params).view(np.int32), p.view(np.int32))
    assert np.array_equal(sums.cpu().numpy(), s)


def values(rows, cols, seed):
    g = np.random.Generator(np.random.PCG64(seed))
    x = g.normal(0, 1, (rows, cols)) * np.exp2(g.integers(-20, 20, (rows, 1))) + g.choice([0.0, 0.0, 30.0, -1e3], (rows, 1))
    return x.astype(np.float32)


@pytest.mark.parametrize("rows,cols", [(1, 1), (7, 127), (9, 128), (5, 129), (3000, 256), (2500, 260), (20000, 500), (9000, 512),
                                       (9001, 516), (5000, 1000), (17, 1024), (33, 1028), (4, 4100), (50, 63),
                                       (50, 64), (50, 97), (40, 31), (41, 32), (42, 33), (30, 65), (70, 200), (60, 257)])
@pytest.mark.parametrize("pad,off", [(0, 0), (4, 0), (3, 1)])
def test_rows(qnn, rows, cols, pad, off):
    check(qnn, values(rows, cols, rows + cols), cols + pad, off, oracle.PER_ROW)


@pytest.mark.parametrize("rows,cols", [(1, 1), (3, 2047), (8, 2048), (9, 2049), (700, 2052), (130, 4099), (5, 16384), (3000, 40),
                                       (1, 100001), (513, 2500), (20001, 57), (15000, 511), (10003, 512),
                                       (3, 8191), (4, 8192), (5, 8193), (600, 2727), (2, 4097), (70000, 17), (90, 63), (90, 65), (4000, 119)])
@pytest.mark.parametrize("pad,off", [(0, 0), (4, 0), (3, 1)])
def test_matrix(qnn, rows, cols, pad, off):
    g = np.random.Generator(np.random.PCG64(rows * 7 + cols))
    check(qnn, (g.normal(0, 0.05, (rows, cols)) + g.choice([0.0, 5.0])).astype(np.float32), cols + pad, off, oracle.PER_MATRIX)


@pytest.mark.parametrize("granularity", [0, 1])
@pytest.mark.parametrize("rows,cols", [(12, 300), (6, 3000)])
@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
def test_non_finite_values_are_reported(qnn, rows, cols, value, granularity):
    x = values(rows, cols, 3)
    for at in ((0, 0), (rows - 1, cols - 1), (rows // 2, cols // 2)):
        bad = x.copy()
        bad[at] = value
        qnn.qnn_quantize(torch.from_numpy(bad).cuda(), granularity)
        assert qnn.device_status() == qnn.QNN_ERR_NONFINITE
    qnn.qnn_quantize(torch.from_numpy(x).cuda(), granularity)
    assert qnn.device_status() == qnn.QNN_OK


# Units whose scale 255 / max|v| is infinite, of every sign and with zeros, among ordinary rows and alone: on each
# kernel's widths.
@pytest.mark.parametrize("form", ["rows", "matrix", "static"])
@pytest.mark.parametrize("cols,pad,off", [(1, 0, 0), (60, 0, 0), (500, 0, 0), (1000, 4, 0), (57, 3, 1), (1500, 4, 0), (2100, 0, 0),
                                          (2101, 0, 0)])
@pytest.mark.parametrize("tiny", [7e-37, 1e-37, 1e-40, 1e-45])
def test_units_of_infinite_scale(qnn, form, cols, pad, off, tiny):
    g = np.random.Generator(np.random.PCG64(cols))
    t = np.float32(tiny)
    mixed = np.where(g.integers(0, 2, (3, cols)) == 1, t, -t).astype(np.float32)
    kinds = [mixed, np.abs(mixed), -np.abs(mixed), mixed * g.integers(0, 2, (3, cols)).astype(np.float32),
             np.abs(mixed) * g.integers(0, 2, (3, cols)).astype(np.float32), -np.abs(mixed) * g.integers(0, 2, (3, cols)).astype(np.float32)]
    kinds = [k + np.float32(0) for k in kinds]  # (no negative zeros: the sign of a range's zero is not pinned)
    if form == "rows":
        x = np.concatenate([np.concatenate([k, values(1, cols, i)]) for i, k in enumerate(kinds)])
        check(qnn, x, cols + pad, off, oracle.PER_ROW)
        return
    for k in kinds:
        check(qnn, k, cols + pad, off, oracle.PER_MATRIX, static=form == "static")


# Frames and states whose units have an infinite scale: the recurrences recover 0 from any of their codes, on each path.
@pytest.mark.parametrize("path,B", [("small", 2), ("persist", 9), ("layerwise", 9), ("tc", 66)])
def test_recurrence_on_units_of_infinite_scale(qnn, path, B, monkeypatch):
    monkeypatch.setenv("QNN_LSTM_PATH", path)
    L, I, H, T = 2, 24, 32, 3
    g = np.random.Generator(np.random.PCG64(B))
    d = oracle.desc(L, I, H, 0, 0, oracle.OUT_NONE)
    params = g.uniform(-0.5, 0.5, oracle.lstm_param_count(d)).astype(np.float32)
    x = g.normal(0, 1, (B, T, I)).astype(np.float32)
    x[:, 0] *= np.float32(1e-38)  # a frame of every sequence, and every frame of some
    x[::2] *= np.float32(1e-38)
    h0, c0 = ((g.normal(0, 1, (L, B, H)) * 1e-39).astype(np.float32) for _ in range(2))
    ref = oracle.lstm_forward(d, params, x, h0=h0, c0=c0, want_h_all=True)
    model = qnn.LstmModel(qnn.lstm_desc(L, I, H), torch.from_numpy(params).cuda())
    hs, cs, ha = torch.from_numpy(h0.copy()).cuda(), torch.from_numpy(c0.copy()).cuda(), torch.empty((L, B, T, H), device="cuda")
    model.forward(torch.from_numpy(x).cuda(), h_state=hs, c_state=cs, h_all=ha)
    assert qnn.device_status() == qnn.QNN_OK
    assert np.array_equal(ha.cpu().numpy(), ref["h_all"]) and np.array_equal(cs.cpu().numpy(), ref["c"])
