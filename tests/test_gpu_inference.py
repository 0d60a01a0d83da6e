"""The network's inference in one kernel, the grouped ends of its training step, and the column
statistics of its rows, at the edges of their tiles."""
import numpy as np
import pytest

from paper_2411_05799_gb300 import npx

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(autouse=True)
def _own_stream():
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        yield
    s.synchronize()


def _layer_by_layer(Ws, bs, x):
    """The same network from the public GEMM: BF16 operands padded to its tiles, one launch a layer."""
    pad = lambda n: (n + 127) // 128 * 128
    M = x.shape[0]
    st = torch.cuda.current_stream().cuda_stream
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    h = torch.zeros(M, pad(x.shape[1]), dtype=torch.bfloat16, device="cuda")
    h[:, :x.shape[1]] = x.to(torch.bfloat16)
    for l, (W, b) in enumerate(zip(Ws, bs)):
        n, k = pad(W.shape[0]), h.shape[1]
        Wp = torch.zeros(n, k, dtype=torch.bfloat16, device="cuda")
        Wp[:W.shape[0], :W.shape[1]] = torch.from_numpy(W).cuda().to(torch.bfloat16)
        bp = torch.zeros(n, device="cuda")
        bp[:len(b)] = torch.from_numpy(b).cuda()
        last = l == len(Ws) - 1
        out = torch.zeros(M, n, dtype=torch.float32 if last else torch.bfloat16, device="cuda")
        ep = npx.GemmEpilogue(mode=npx.EPI_BIAS if last else npx.EPI_BIAS_GELU, bias=bp.data_ptr(),
                              **({"outf": out.data_ptr(), "ldf": n} if last else {"out": out.data_ptr(), "ldo": n}))
        npx.gemm_bf16(h.data_ptr(), Wp.data_ptr(), M, n, k, ep, err.data_ptr(), stream=st)
        torch.cuda.synchronize()
        h = out
    assert int(err.item()) == 0
    return h[:, :Ws[-1].shape[0]]


@pytest.mark.parametrize("M,n_in,hidden,layers,n_out", [
    (128, 271, 512, 4, 247),      # one tile
    (128 * 153, 271, 512, 4, 247),    # one tile more than there are SMs
    (384, 1, 128, 1, 1),          # one block, one input, one output
    (256, 64, 256, 7, 129),       # eight layers, one block each, an odd output width
    (640, 300, 384, 2, 300),      # blocks of 256 and 128, outputs in two blocks
    (128 * 305, 512, 512, 1, 512),    # the widest, three tiles on some SMs
    (256, 40, 640, 2, 30),        # too wide for one kernel
    (256, 40, 128, 8, 30),        # too deep for one kernel
])
def test_inference_equals_the_layers_one_by_one(M, n_in, hidden, layers, n_out):
    """Same operands, products in the same order, same roundings: equal bit for bit."""
    rng = np.random.default_rng(M + hidden)
    sizes = [n_in] + [hidden] * layers + [n_out]
    Ws = [rng.normal(0, np.sqrt(2 / i), (o, i)).astype(np.float32) for i, o in zip(sizes[:-1], sizes[1:])]
    bs = [rng.normal(0, 0.1, o).astype(np.float32) for o in sizes[1:]]
    net = npx.MLP(n_in, n_out, n_hidden=hidden, n_hidden_layers=layers, max_batch=M,
                  stream=torch.cuda.current_stream().cuda_stream)
    net.set_params(Ws, bs)
    x = torch.from_numpy(rng.normal(0, 1, (M, n_in)).astype(np.float32)).cuda()
    y = torch.full((M + 1, n_out), float("nan"), device="cuda")
    for _ in range(2):
        net.forward(x.data_ptr(), y.data_ptr(), M)
    torch.cuda.synchronize()
    assert torch.equal(y[:M], _layer_by_layer(Ws, bs, x))
    assert torch.isnan(y[M]).all()          # nothing past the last row
    if n_out <= n_in:                       # outputs over the inputs
        net.forward(x.data_ptr(), x.data_ptr(), M)
        torch.cuda.synchronize()
        assert torch.equal(x.reshape(-1)[:M * n_out].reshape(M, n_out), y[:M])


@pytest.mark.parametrize("rows,cols", [(1, 1), (7, 3), (2047, 36), (2048, 37), (4097, 72), (999, 73), (1000, 144),
                                       (5000, 145), (3001, 271)])
def test_column_moments(rows, cols):
    """FP64 sums: n terms in any order stay within n 2^-53 sum |term| of the exact sum (here against
    numpy's, itself within a few 2^-53); they add to what is there and repeat bit for bit."""
    g = torch.Generator("cuda").manual_seed(rows)
    X = torch.randn(rows, cols, device="cuda", generator=g) * 10.0 ** (torch.arange(cols, device="cuda") % 5 - 2) + 1.0
    st = torch.cuda.current_stream().cuda_stream
    got = []
    for _ in range(2):
        s = torch.full((2, cols), 0.5, dtype=torch.float64, device="cuda")
        npx.column_moments(X.data_ptr(), rows, cols, s[0].data_ptr(), s[1].data_ptr(), st)
        torch.cuda.synchronize()
        got.append(s.cpu().numpy())
    np.testing.assert_array_equal(got[0], got[1])
    h = X.cpu().numpy().astype(np.float64)
    for k, v in enumerate((h, h * h)):
        exact = np.array([np.sum(v[:, c].astype(np.longdouble)) for c in range(cols)], dtype=np.float64)
        bound = (rows + 2) * 2.0 ** -53 * (np.abs(v).sum(0) + 0.5) * 1.01
        assert (np.abs(got[0][k] - 0.5 - exact) <= bound).all()


def test_column_moments_of_infinities_and_nan():
    X = torch.ones(3000, 5, device="cuda")
    X[5, 1], X[2999, 2], X[7, 3], X[8, 3] = float("inf"), float("nan"), float("inf"), float("-inf")
    s = torch.zeros(2, 5, dtype=torch.float64, device="cuda")
    npx.column_moments(X.data_ptr(), 3000, 5, s[0].data_ptr(), s[1].data_ptr(), torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    a, q = s.cpu().numpy()
    assert a[0] == 3000 and a[1] == np.inf and np.isnan(a[2]) and np.isnan(a[3]) and a[4] == 3000
    assert q[1] == np.inf and np.isnan(q[2]) and q[3] == np.inf


@pytest.mark.parametrize("M,n_in,hidden,layers,n_out", [(128, 3, 128, 1, 2), (1152, 271, 256, 2, 129),
                                                        (2048, 40, 128, 17, 30)])
def test_training_step(M, n_in, hidden, layers, n_out):
    """One launch for what is left of the gradients and one for Adam, up to sixteen layers at a time
    (17 hidden layers take two): bias gradients against FP64 sums of the network's own BF16 output
    gradients where those are known (the last layer), weights after Adam's first step against its
    formula on the gradients read back, element by element."""
    rng = np.random.default_rng(M)
    sizes = [n_in] + [hidden] * layers + [n_out]
    Ws = [rng.normal(0, np.sqrt(2 / i), (o, i)).astype(np.float32) for i, o in zip(sizes[:-1], sizes[1:])]
    bs = [rng.normal(0, 0.1, o).astype(np.float32) for o in sizes[1:]]
    net = npx.MLP(n_in, n_out, n_hidden=hidden, n_hidden_layers=layers, max_batch=M, lr=1e-3,
                  stream=torch.cuda.current_stream().cuda_stream)
    net.set_params(Ws, bs)
    x = torch.from_numpy(rng.normal(0, 1, (M, n_in)).astype(np.float32)).cuda()
    t = torch.from_numpy(rng.normal(0, 1, (M, n_out)).astype(np.float32)).cuda()
    y = torch.zeros(M, n_out, device="cuda")
    loss = torch.zeros(1, device="cuda")
    net.forward(x.data_ptr(), y.data_ptr(), M)
    net.backward(x.data_ptr(), t.data_ptr(), M, loss.data_ptr())
    gWs, gbs = net.get_grads()
    net.adam_step()
    torch.cuda.synchronize()
    W1, b1 = net.get_params()
    # the last layer's bias gradient: the column sums of BF16(2 (y - t) / M); M FP32 terms in any order
    # stay within M 2^-24 of the sum of their magnitudes
    inv = torch.tensor(1.0, device="cuda") / M
    g = (2.0 * (y - t) * inv).to(torch.bfloat16).double().cpu().numpy()
    assert (np.abs(gbs[-1] - g.sum(0)) <= M * 2.0 ** -24 * np.abs(g).sum(0)).all()
    assert all(np.isfinite(a).all() for a in gWs + gbs)
    # Adam's first step: m / (1 - 0.9) = g, v / (1 - 0.999) = g^2, so p - lr g / (|g| + eps); the FP32
    # 1 - 0.9 and 1 - 0.999 are off by up to 2^-24 / 0.001 relative
    for p0, p1, gr in zip(Ws + bs, W1 + b1, gWs + gbs):
        step = 1e-3 * gr.astype(np.float64) / (np.abs(gr.astype(np.float64)) + 1e-8)
        assert (np.abs(p1 - (p0 - step)) <= 2.0 ** -23 * (np.abs(p0) + 1e-3) + 1e-3 * 2e-4).all()
    # and the BF16 copies the next pass reads are the new weights': the forward pass uses them
    net.forward(x.data_ptr(), y.data_ptr(), M)
    torch.cuda.synchronize()
    assert torch.equal(y, _layer_by_layer(W1, b1, x))
    # (the transposes too: two networks with the same parameters give the same gradients)
    other = npx.MLP(n_in, n_out, n_hidden=hidden, n_hidden_layers=layers, max_batch=M,
                    stream=torch.cuda.current_stream().cuda_stream)
    other.set_params(W1, b1)
    for n in (net, other):
        n.backward(x.data_ptr(), t.data_ptr(), M, loss.data_ptr())
    for a, b in zip(sum(net.get_grads(), []), sum(other.get_grads(), [])):
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("M,n_in,hidden,layers,n_out", [(128, 3, 128, 1, 2), (1152, 271, 256, 2, 129),
                                                        (2048, 200, 256, 10, 300), (192 * 128, 40, 128, 2, 30)])
def test_weight_gradients_together(M, n_in, hidden, layers, n_out):
    """The layers' weight gradients come from as few launches as their widths allow (eight products
    at most in one, 256 columns a tile apart from 128): each against the FP64 product of the BF16
    arrays, taken by torch through the network's own formulas.  A BF16 array may differ from the
    network's where an FP32 sum rounds the other way (half an ulp, 2^-9 of an element), and each of
    the two arrays of a product passes through at most 2 (layers + 1) roundings: 2 (layers + 1) 2^-8
    of the gradient's norm covers both."""
    rng = np.random.default_rng(M + layers)
    sizes = [n_in] + [hidden] * layers + [n_out]
    Ws = [rng.normal(0, np.sqrt(2 / i), (o, i)).astype(np.float32) for i, o in zip(sizes[:-1], sizes[1:])]
    bs = [rng.normal(0, 0.1, o).astype(np.float32) for o in sizes[1:]]
    net = npx.MLP(n_in, n_out, n_hidden=hidden, n_hidden_layers=layers, max_batch=M,
                  stream=torch.cuda.current_stream().cuda_stream)
    net.set_params(Ws, bs)
    x = torch.from_numpy(rng.normal(0, 1, (M, n_in)).astype(np.float32)).cuda()
    t = torch.from_numpy(rng.normal(0, 1, (M, n_out)).astype(np.float32)).cuda()
    loss = torch.zeros(1, device="cuda")
    for _ in range(2):   # (the second pass right behind the first: nothing of it may be read early)
        net.backward(x.data_ptr(), t.data_ptr(), M, loss.data_ptr())
    torch.cuda.synchronize()
    gWs, gbs = net.get_grads()
    r = lambda a: a.to(torch.bfloat16).double()
    W = [r(torch.from_numpy(w).cuda()) for w in Ws]
    b = [torch.from_numpy(v).cuda().double() for v in bs]
    X, Z = [r(x)], []
    for l in range(layers):
        z = X[-1] @ W[l].T + b[l]
        Z.append(r(z))
        X.append(r(torch.nn.functional.gelu(z, approximate="tanh")))
    d = r(2.0 * (X[-1] @ W[-1].T + b[-1] - t.double()) / M)
    for l in range(layers, -1, -1):
        ref = d.T @ X[l]
        err = (torch.from_numpy(gWs[l]).cuda().double() - ref).norm() / ref.norm()
        assert float(err) <= 2 * (layers + 1) * 2.0 ** -8, (l, float(err))
        if l:
            z = Z[l - 1].clone().requires_grad_(True)
            dg, = torch.autograd.grad(torch.nn.functional.gelu(z, approximate="tanh").sum(), z)
            d = r((d @ W[l]) * dg)


@pytest.mark.parametrize("mode", [npx.EPI_BIAS, npx.EPI_BIAS_GELU, npx.EPI_DGELU])
@pytest.mark.parametrize("ldt, off", [(640, 0), (640, 1), (641, 0), (641, 1), (642, 2)])
def test_transposed_output_on_any_address(mode, ldt, off):
    """C^T goes out two rows to a store where its columns start on 4 bytes, one row otherwise: the same
    values either way, nothing written beside them, and the transpose of the row-major output."""
    M, N, K = 640, 384, 128
    g = torch.Generator(device="cpu").manual_seed(ldt + off)
    A = torch.randn(M, K, generator=g).to(torch.bfloat16).cuda()
    B = torch.randn(N, K, generator=g).to(torch.bfloat16).cuda()
    b = torch.randn(N, generator=g).cuda()
    z = torch.randn(M, N, generator=g).to(torch.bfloat16).cuda()
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    out = torch.zeros(M, N, dtype=torch.bfloat16, device="cuda")
    zs = torch.zeros(M, N, dtype=torch.bfloat16, device="cuda")
    flat = torch.full((N * ldt + off,), 7.0, dtype=torch.bfloat16, device="cuda")
    ep = npx.GemmEpilogue(mode=mode, bias=b.data_ptr() if mode != npx.EPI_DGELU else None, out=out.data_ptr(), ldo=N,
                          outT=flat.data_ptr() + 2 * off, ldt=ldt,
                          zsave=zs.data_ptr() if mode == npx.EPI_BIAS_GELU else None, ldz=N, zin=z.data_ptr(), ldzi=N)
    npx.gemm_bf16(A.data_ptr(), B.data_ptr(), M, N, K, ep, err.data_ptr())
    torch.cuda.synchronize()
    assert int(err.item()) == 0
    T = flat[off:].reshape(N, ldt)
    assert torch.equal(T[:, :M], out.T)
    assert (flat[:off] == 7.0).all() and (T[:, M:] == 7.0).all()
    if mode == npx.EPI_BIAS_GELU:   # the pre-activations: FP32 sums of K products, rounded to BF16
        ref = A.double() @ B.double().T + b.double()
        assert ((zs.double() - ref).abs() <= 2.0 ** -8 * ref.abs() + 1e-4).all()
