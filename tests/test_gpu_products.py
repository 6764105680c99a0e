"""The product kernels at the edges of their tiles: the streaming integer-MMA kernel over every
number of A-row groups, ragged rows, ragged reductions and row alignments (16, 4 and 1 bytes), the
tensor-core product's outputs, and the product from the codes at its own edges."""
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


def gpu(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def strided(a, ld, off):
    """The code matrix on the device with `ld` bytes between rows, starting `off` bytes into its
    buffer; the bytes between and after the rows are nonzero codes that must not be summed."""
    rows, cols = a.shape
    buf = torch.full((off + rows * ld,), 77, dtype=torch.uint8, device="cuda")
    v = buf[off:].reshape(rows, ld)[:, :cols]
    v.copy_(gpu(a))
    return v


# M around the 8-row groups of A (1, 2, 4 and 8 per block), N around 16 and 32 rows of W, K around
# 16 codes, the 64-code chunk and the 8 warps' round of chunks
@pytest.mark.parametrize("M,N,K", [(1, 1, 1), (1, 16, 64), (1, 2000, 500), (1, 33, 4097), (7, 17, 15), (8, 31, 513),
                                   (9, 15, 63), (16, 100, 1000), (17, 16, 65), (32, 130, 2049), (33, 31, 16),
                                   (64, 33, 511), (65, 64, 129), (100, 2000, 500), (127, 96, 8192), (2, 64, 33025)])
@pytest.mark.parametrize("pad,off", [(None, 0), (0, 0), (4, 4), (3, 1)])
def test_few_rows_bit_exact(qnn, M, N, K, pad, off, monkeypatch):
    monkeypatch.setenv("QNN_QGEMM", "imma")
    g = np.random.Generator(np.random.PCG64(M * 31 + N * 7 + K))
    A = g.normal(0.1, 1.0, (M, K)).astype(np.float32)
    nb = 4 if N % 4 == 0 else 1
    Ws = [g.uniform(-s, s, (N // nb, K)).astype(np.float32) for s in np.linspace(0.05, 0.4, nb)]
    ga = oracle.PER_ROW if M % 2 else oracle.PER_MATRIX
    ca, pa, ra = oracle.quantize(A, ga)
    parts = [oracle.quantize(w, oracle.PER_MATRIX) for w in Ws]
    cw, pw, cs = (np.concatenate([p[i] for p in parts]) for i in range(3))
    bias = g.normal(0, 1, N).astype(np.float32) if K % 2 else None
    ref = oracle.qmatmul(ca, pa, ga, cw, pw, n_blocks=nb, bias=bias)
    ld = (K + 15) // 16 * 16 if pad is None else (K + 3) // 4 * 4 + pad if pad == 4 else K + pad
    Y, acc = qnn.qnn_qmatmul(strided(ca, ld, off), qnn.params_tensor(pa), ga, gpu(ra), strided(cw, ld, off),
                             qnn.params_tensor(pw), gpu(cs), n_blocks=nb, bias=None if bias is None else gpu(bias),
                             want_acc=True)
    assert qnn.device_status() == qnn.QNN_OK
    assert np.array_equal(acc.cpu().numpy(), ref["acc"])
    assert np.array_equal(Y.cpu().numpy(), ref["y"])


# The float output layer on each of its tiles (32, 64 and 128 rows and classes, chosen by the number of
# tiles), with ragged rows and classes and K not a multiple of 4 or of 16, against the oracle's fp64
# sums within the fp32 dot-product bound (parity.float_logit_bound).
@pytest.mark.parametrize("B,T,H,C", [(5, 3, 50, 33), (7, 5, 64, 300), (70, 9, 50, 1999), (64, 10, 36, 2000),
                                     (65, 20, 49, 2001), (100, 17, 64, 1300)])
def test_float_output_layer_tiles(qnn, B, T, H, C):
    import parity
    from paper_1607_04683_gb300 import inputs
    wl = inputs.LstmWorkload("float", seed=3, num_layers=1, input_dim=12, hidden=H, proj=0, num_classes=C, batch=B,
                             frames=T, w_range=0.3, forget_bias=1.0, output_mode=2, out_w_range=0.5)
    params, x = wl.make()
    model = qnn.LstmModel(qnn.lstm_desc(1, 12, H, 0, C, qnn.OUT_FLOAT), gpu(params))
    lg = torch.full((B, T, C), float("nan"), device="cuda")
    y = model.forward(gpu(x), logits=lg)
    assert qnn.device_status() == qnn.QNN_OK
    ref = oracle.lstm_forward(oracle.desc(1, 12, H, 0, C, oracle.OUT_FLOAT), params, x, want_h_all=True,
                              want_logits=True)
    parity.check_logits(lg.cpu().numpy(), ref["logits"], 2, ref["h_all"][0], wl.out_weights(params))
    parity.check_posteriors(y.cpu().numpy(), ref["y"])


# The tensor-core product's outputs without raw sums: K <= 1024 stores them by TMA from staging buffers
# (whole units, ragged rows and columns, rows further apart than N, unaligned rows by plain stores), longer K
# whole blocks of 32 columns in 32-bit sums; offsets beyond the fp32 and the 32-bit forms take the others.
@pytest.mark.parametrize("bn", ["64", "128", "256", "512"])
@pytest.mark.parametrize("M,N,K,pad", [(1, 8, 1, 0), (33, 64, 64, 0), (128, 256, 64, 4), (130, 260, 100, 0), (257, 2000, 500, 8),
                                       (200, 136, 1000, 1), (384, 512, 1024, 0), (129, 260, 1025, 0), (257, 320, 3000, 4), (140, 261, 1100, 0),
                                       (260, 515, 2100, 1), (161, 163, 300, 0)])
@pytest.mark.parametrize("shift", [0.0, 20.0, 3000.0])
def test_tensor_core_outputs(qnn, M, N, K, pad, bn, shift, monkeypatch):
    monkeypatch.setenv("QNN_QGEMM", "tc")
    monkeypatch.setenv("QNN_TC_BN", bn)
    g = np.random.Generator(np.random.PCG64(M + N + K))
    A = (g.normal(0.1, 1.0, (M, K)) + shift).astype(np.float32)
    nb = 4 if N % 4 == 0 else 1
    Ws = [g.uniform(-s, s, (N // nb, K)).astype(np.float32) for s in np.linspace(0.05, 0.4, nb)]
    ga = oracle.PER_ROW if M % 2 else oracle.PER_MATRIX
    ca, pa, ra = oracle.quantize(A, ga)
    parts = [oracle.quantize(w, oracle.PER_MATRIX) for w in Ws]
    cw, pw, cs = (np.concatenate([p[i] for p in parts]) for i in range(3))
    bias = g.normal(0, 1, N).astype(np.float32) if K % 2 == 0 else None
    ref = oracle.qmatmul(ca, pa, ga, cw, pw, n_blocks=nb, bias=bias)
    out = torch.full((M + 1, N + pad), 7.0, device="cuda")
    qnn.qnn_qmatmul(gpu(ca), qnn.params_tensor(pa), ga, gpu(ra), gpu(cw), qnn.params_tensor(pw), gpu(cs), n_blocks=nb,
                    bias=None if bias is None else gpu(bias), out=out[:M, :N])
    assert qnn.device_status() == qnn.QNN_OK
    assert np.array_equal(out[:M, :N].cpu().numpy(), ref["y"])
    assert bool((out[M:] == 7.0).all()) and bool((out[:, N:] == 7.0).all())


# The product from the codes: rows of A around its 64 and 128 columns, rows of W around 128, K around 16 codes,
# a stage of 128 codes (one and two k-blocks of it), the ring's three stages with two of loads ahead, chunks of
# eight stages (drained a stage into the next; a last chunk of one stage, or of part of one), every row shift, raw
# sums, sums of 32 and of 64 bits.
@pytest.mark.parametrize("M,N,K", [(1, 1, 40), (5, 6, 7), (63, 127, 15), (64, 128, 16), (65, 129, 17), (100, 260, 63), (129, 2000, 64),
                                   (130, 500, 65), (200, 9000, 127), (128, 20000, 193), (128, 130, 256), (129, 136, 321),
                                   (300, 300, 1000), (128, 64, 1024), (130, 132, 1025), (96, 128, 1088), (70, 200, 1153),
                                   (128, 14600, 1217), (128, 129, 2048), (128, 128, 2113), (66, 65, 3300), (64, 33, 33025),
                                   (130, 1500, 1500), (40, 300, 1023), (128, 1100, 1025), (300, 700, 2050)])
@pytest.mark.parametrize("pad,off,shift", [(None, 0, 0.0), (0, 0, 20.0), (4, 4, 3000.0), (3, 1, 0.0), (6, 15, 0.0)])
def test_codes_bit_exact(qnn, M, N, K, pad, off, shift, monkeypatch):
    monkeypatch.setenv("QNN_QGEMM", "codes")
    g = np.random.Generator(np.random.PCG64(M * 31 + N * 7 + K))
    A = (g.normal(0.1, 1.0, (M, K)) + shift).astype(np.float32)
    nb = 4 if N % 4 == 0 else 1
    Ws = [g.uniform(-s, s, (N // nb, K)).astype(np.float32) for s in np.linspace(0.05, 0.4, nb)]
    ga = oracle.PER_ROW if M % 2 else oracle.PER_MATRIX
    ca, pa, ra = oracle.quantize(A, ga)
    parts = [oracle.quantize(w, oracle.PER_MATRIX) for w in Ws]
    cw, pw, cs = (np.concatenate([p[i] for p in parts]) for i in range(3))
    bias = g.normal(0, 1, N).astype(np.float32) if K % 2 else None
    ref = oracle.qmatmul(ca, pa, ga, cw, pw, n_blocks=nb, bias=bias)
    ld = (K + 15) // 16 * 16 if pad is None else (K + 3) // 4 * 4 + pad if pad == 4 else K + pad
    out = torch.full((M + 1, N + 3), 7.0, device="cuda")
    _, acc = qnn.qnn_qmatmul(strided(ca, ld, off), qnn.params_tensor(pa), ga, gpu(ra), strided(cw, ld, off),
                             qnn.params_tensor(pw), gpu(cs), n_blocks=nb, bias=None if bias is None else gpu(bias),
                             want_acc=True, out=out[:M, :N])
    assert qnn.device_status() == qnn.QNN_OK
    assert np.array_equal(acc.cpu().numpy(), ref["acc"])
    assert np.array_equal(out[:M, :N].cpu().numpy(), ref["y"])
    assert bool((out[M:] == 7.0).all()) and bool((out[:, N:] == 7.0).all())


# Raw sums beside the tensor-core product's outputs for K <= 1024: tiles of 64 and 128 columns, rows of sums of any
# alignment (N odd), ragged tiles, columns of several weight units, outputs by TMA and by plain stores.
@pytest.mark.parametrize("bn", ["64", "128"])
@pytest.mark.parametrize("M,N,K,nb,pad", [(1, 8, 1, 1, 0), (33, 64, 64, 4, 0), (130, 261, 100, 1, 0), (257, 2000, 500, 4, 8), (200, 135, 1000, 3, 1),
                                          (384, 513, 1024, 1, 0), (129, 2001, 32, 1, 0)])
def test_tensor_core_raw_sums(qnn, M, N, K, nb, pad, bn, monkeypatch):
    monkeypatch.setenv("QNN_QGEMM", "tc")
    monkeypatch.setenv("QNN_TC_BN", bn)
    g = np.random.Generator(np.random.PCG64(M + N + K))
    ca, pa, ra = oracle.quantize(g.uniform(0, 1, (M, K)).astype(np.float32), oracle.PER_ROW)
    parts = [oracle.quantize(g.uniform(-s, s, (N // nb, K)).astype(np.float32), oracle.PER_MATRIX) for s in np.linspace(0.05, 0.4, nb)]
    cw, pw, cs = (np.concatenate([p[i] for p in parts]) for i in range(3))
    ref = oracle.qmatmul(ca, pa, oracle.PER_ROW, cw, pw, n_blocks=nb)
    out = torch.full((M + 1, N + pad), 7.0, device="cuda")
    _, acc = qnn.qnn_qmatmul(gpu(ca), qnn.params_tensor(pa), oracle.PER_ROW, gpu(ra), gpu(cw), qnn.params_tensor(pw), gpu(cs),
                             n_blocks=nb, want_acc=True, out=out[:M, :N])
    assert qnn.device_status() == qnn.QNN_OK
    assert np.array_equal(acc.cpu().numpy(), ref["acc"]) and np.array_equal(out[:M, :N].cpu().numpy(), ref["y"])
    assert bool((out[M:] == 7.0).all()) and bool((out[:, N:] == 7.0).all())


# One and two tiles share their reductions between the blocks of a cluster: `parts` of them with K, the last one of
# one stage, of less than a stage or of an odd number of k-blocks, and chunks that end inside a part.
@pytest.mark.parametrize("M,N", [(33, 128), (64, 250), (70, 100)])
@pytest.mark.parametrize("K,parts", [(1023, 2), (1024, 2), (1600, 3), (1665, 3), (2049, 4), (2600, 5), (2561, 5), (4096, 8), (4100, 7), (8200, 8), (33025, 8)])
@pytest.mark.parametrize("pad,off", [(None, 0), (0, 0), (3, 1)])
def test_codes_shared_reductions(qnn, M, N, K, parts, pad, off, monkeypatch):
    monkeypatch.setenv("QNN_QGEMM", "codes")
    steps = -(-K // 128)  # stages; the rule of launch_codes where SMs are plenty
    splits = max(1, min(8, steps // 4))
    assert -(-steps // -(-steps // splits)) == parts
    g = np.random.Generator(np.random.PCG64(M + N + K))
    ca, pa, ra = oracle.quantize(g.normal(0.1, 1.0, (M, K)).astype(np.float32), oracle.PER_ROW)
    cw, pw, cs = oracle.quantize(g.normal(0.0, 1.0, (N, K)).astype(np.float32), oracle.PER_MATRIX)
    ref = oracle.qmatmul(ca, pa, oracle.PER_ROW, cw, pw)
    ld = (K + 15) // 16 * 16 if pad is None else K + pad
    qnn.profile_read()
    qnn.profile_enable(True)
    Y, acc = qnn.qnn_qmatmul(strided(ca, ld, off), qnn.params_tensor(pa), oracle.PER_ROW, gpu(ra), strided(cw, ld, off),
                             qnn.params_tensor(pw), gpu(cs), want_acc=True)
    qnn.profile_enable(False)
    assert "qgemm_codes_split" in qnn.profile_read()
    assert qnn.device_status() == qnn.QNN_OK
    assert np.array_equal(acc.cpu().numpy(), ref["acc"]) and np.array_equal(Y.cpu().numpy(), ref["y"])


# Operands too small to hold one aligned unit take another path than the one the sizes ask for.
@pytest.mark.parametrize("M,N,K", [(130, 1, 1), (200, 2, 15), (129, 1, 30), (128, 1, 31)])
@pytest.mark.parametrize("off", [0, 1, 15])
def test_few_codes(qnn, M, N, K, off):
    g = np.random.Generator(np.random.PCG64(M + K))
    ca, pa, ra = oracle.quantize(g.normal(0.1, 1.0, (M, K)).astype(np.float32), oracle.PER_ROW)
    cw, pw, cs = oracle.quantize(g.normal(0.0, 1.0, (N, K)).astype(np.float32), oracle.PER_MATRIX)
    ref = oracle.qmatmul(ca, pa, oracle.PER_ROW, cw, pw)
    Y, acc = qnn.qnn_qmatmul(strided(ca, K, off), qnn.params_tensor(pa), oracle.PER_ROW, gpu(ra), strided(cw, K, off),
                             qnn.params_tensor(pw), gpu(cs), want_acc=True)
    assert qnn.device_status() == qnn.QNN_OK
    assert np.array_equal(acc.cpu().numpy(), ref["acc"]) and np.array_equal(Y.cpu().numpy(), ref["y"])


# Centering both operands, rows of any alignment: around 8 codes, whole and ragged rows, the first and last
# codes of a matrix, more than one round of a thread's groups.
@pytest.mark.parametrize("M,N,K", [(130, 70, 1), (130, 70, 7), (129, 65, 8), (131, 64, 9), (200, 3, 23), (150, 150, 65), (140, 90, 1030),
                                   (9000, 2000, 517)])
@pytest.mark.parametrize("pad,off", [(0, 0), (0, 1), (3, 7), (8, 8)])
def test_centered_operands(qnn, M, N, K, pad, off, monkeypatch):
    monkeypatch.setenv("QNN_QGEMM", "tc")
    g = np.random.Generator(np.random.PCG64(M + N + K))
    ca, pa, ra = oracle.quantize(g.normal(0.1, 1.0, (M, K)).astype(np.float32), oracle.PER_ROW)
    cw, pw, cs = oracle.quantize(g.normal(0.0, 1.0, (N, K)).astype(np.float32), oracle.PER_MATRIX)
    ref = oracle.qmatmul(ca, pa, oracle.PER_ROW, cw, pw)
    _, acc = qnn.qnn_qmatmul(strided(ca, K + pad, off), qnn.params_tensor(pa), oracle.PER_ROW, gpu(ra), strided(cw, K + pad, off),
                             qnn.params_tensor(pw), gpu(cs), want_acc=True)
    assert qnn.device_status() == qnn.QNN_OK
    assert np.array_equal(acc.cpu().numpy(), ref["acc"])


# Gate tiles of 32, 64 and 128 columns in a wavefront of layers, by the tiles of all layers.
@pytest.mark.parametrize("L,H,P,B", [(2, 512, 128, 70), (3, 512, 64, 130), (3, 520, 0, 260), (2, 1024, 128, 300)])
def test_gate_tiles_of_a_wavefront(qnn, L, H, P, B, monkeypatch):
    from paper_1607_04683_gb300 import inputs
    monkeypatch.setenv("QNN_LSTM_PATH", "tc")
    wl = inputs.LstmWorkload("wave", seed=L + H + B, num_layers=L, input_dim=20, hidden=H, proj=P, num_classes=0, batch=B,
                             frames=3, w_range=0.08, forget_bias=1.0, output_mode=0)
    params, x = wl.make()
    model = qnn.LstmModel(qnn.lstm_desc(L, 20, H, P, 0), gpu(params))
    y = model.forward(gpu(x))
    assert qnn.device_status() == qnn.QNN_OK
    b = [0, 63, B // 2, B - 1]
    ref = oracle.lstm_forward(oracle.desc(L, 20, H, P, 0, oracle.OUT_NONE), params, np.ascontiguousarray(x[b]), want_h_all=True)
    assert np.array_equal(y.cpu().numpy()[b], ref["h_all"][-1])
