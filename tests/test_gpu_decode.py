"""GPU parity of the decode path (few tokens, weights streamed once) against the CPU oracle.
When the row tiles alone fill the GPU the kernel adds each output's blocks in ascending order with
one fp32 rounding per block and must equal the oracle's sequential-fp32 result bit for bit; when K
is cut over warps (single small layers) the result must stay within 1e-5 * S of the exact value."""
import numpy as np
import pytest
import torch

from oracle import mx_oracle as orc
from paper_2307_15517_b200 import synth

pytestmark = pytest.mark.gpu
TOL = 1e-5


@pytest.fixture(scope="module")
def mxb():
    from paper_2307_15517_b200 import binding
    return binding


def _layer(mxb, T, K, N, seed, wa=8, ww=4, with_bias=False, heavy=False):
    x = synth.student_t_activations(T, K, seed) if heavy else synth.decode_activations(T, K, seed)
    w = synth.gaussian_weights(N, K, seed + 1)
    bias = synth.gaussian_weights(1, N, seed + 2, std=1.0)[0] if with_bias else None
    fa, fw = mxb.MxFormat(32, wa), mxb.MxFormat(32, ww)
    qa, ea, _ = orc.quantize(x.numpy(), 32, wa)
    qw, ew, _ = orc.quantize(w.numpy(), 32, ww)
    dev = dict(x=x.cuda(), fa=fa, fw=fw, N=N, bias=None if bias is None else bias.cuda(),
               w_mant=torch.from_numpy(orc.pack(qw, ww)).cuda(), w_exp=torch.from_numpy(ew).cuda(),
               y=torch.full((T, N), -5.0, device="cuda"))
    ref = dict(qa=qa, ea=ea, qw=qw, ew=ew, wa=wa, ww=ww, bias=None if bias is None else bias.numpy())
    return dev, ref


def _oracle(ref):
    return orc.gemm(ref["qa"], ref["ea"], ref["wa"], ref["qw"], ref["ew"], ref["ww"], 32, bias=ref["bias"])


@pytest.mark.parametrize("T", (1, 4, 8, 16))
@pytest.mark.parametrize("shape", [(1024, 512), (4096, 272), (128, 40)])
def test_stream_single_layer_within_tolerance(mxb, T, shape):
    K, N = shape
    dev, ref = _layer(mxb, T, K, N, seed=T + K, with_bias=True, heavy=True)
    y_ref, y_seq, S = _oracle(ref)
    y = mxb.mx_linear(dev["x"], dev["fa"], dev["w_mant"], dev["w_exp"], dev["fw"], N, bias=dev["bias"],
                      y=dev["y"], algo=mxb.MX_ALGO_STREAM)
    err = np.abs(y.cpu().numpy().astype(np.float64) - y_ref)
    assert (err <= TOL * S + 1e-37).all(), float((err / np.maximum(S, 1e-300)).max())
    # AUTO may cut K over a cluster; these sums are exact in any order
    y2 = mxb.mx_linear(dev["x"], dev["fa"], dev["w_mant"], dev["w_exp"], dev["fw"], N, bias=dev["bias"])
    assert torch.equal(y, y2)


@pytest.mark.parametrize("T,n_layers,K", [(1, 20, 256), (4, 20, 256), (16, 10, 256),
                                          (4, 20, 512), (16, 20, 1024), (1, 20, 1536)])
def test_grouped_launch_is_bit_exact_against_sequential_oracle(mxb, T, n_layers, K):
    """Enough row tiles to fill the GPU without cutting K: ascending fp32 block sums, exactly.
    K = 256 takes the MMA kernel in partial steps, K % 512 == 0 in whole ones or, with one token, the row-per-lane kernel."""
    N = 4096
    layers, refs = [], []
    for i in range(n_layers):
        dev, ref = _layer(mxb, T, K, N, seed=100 * T + 3 * i, wa=(8, 6, 4)[i % 3], ww=(4, 3, 2)[i % 3],
                          with_bias=(i % 2 == 0))
        if i % 4 == 1:                          # layers sharing one activation tensor (q, k, v)
            dev["x"], dev["fa"] = layers[-1]["x"], layers[-1]["fa"]
            ref["qa"], ref["ea"], ref["wa"] = refs[-1]["qa"], refs[-1]["ea"], refs[-1]["wa"]
        layers.append(dev)
        refs.append(ref)
    args = mxb.make_linear_args(layers)
    mxb.mx_linear_grouped(args)
    assert mxb.mx_poll_status() == 0
    for dev, ref in zip(layers, refs):
        y_ref, y_seq, S = _oracle(ref)
        assert np.array_equal(dev["y"].cpu().numpy(), y_seq)


def test_stream_mixed_layer_shapes_and_nonfinite(mxb):
    """Different N and K per layer, a ragged last row tile, a poisoned weight and token block."""
    specs = [(4, 512, 1000), (4, 1024, 48), (3, 128, 4096), (4, 512, 1000)]
    layers, refs = [], []
    for i, (T, K, N) in enumerate(specs):
        dev, ref = _layer(mxb, T, K, N, seed=50 + i, with_bias=(i == 1))
        layers.append(dev)
        refs.append(ref)
    refs[2]["ew"][7, 1] = 255
    layers[2]["w_exp"] = torch.from_numpy(refs[2]["ew"]).cuda()
    x3 = layers[3]["x"].clone()
    x3[1, 40] = float("inf")
    layers[3]["x"] = x3
    refs[3]["qa"], refs[3]["ea"], _ = orc.quantize(x3.cpu().numpy(), 32, 8)
    mxb.mx_linear_grouped(mxb.make_linear_args(layers))
    for dev, ref in zip(layers, refs):
        y_ref, y_seq, S = _oracle(ref)
        y = dev["y"].cpu().numpy()
        assert np.array_equal(np.isnan(y), np.isnan(y_ref))
        ok = ~np.isnan(y_ref)
        assert (np.abs(y[ok].astype(np.float64) - y_ref[ok]) <= TOL * S[ok] + 1e-37).all()
    assert np.isnan(layers[2]["y"][:, 7].cpu().numpy()).all()
    assert np.isnan(layers[3]["y"][1].cpu().numpy()).all() and not np.isnan(layers[3]["y"][0].cpu().numpy()).any()


def test_decode_shapes_sampled(mxb):
    """The decode configuration's own shapes (4096 -> 4096 and 4096 -> 11008, 16 tokens):
    every output of 64 sampled weight rows against the oracle."""
    for N in (4096, 11008):
        dev, ref = _layer(mxb, 16, 4096, N, seed=N)
        y = mxb.mx_linear(dev["x"], dev["fa"], dev["w_mant"], dev["w_exp"], dev["fw"], N, y=dev["y"])
        rows = np.random.default_rng(N).choice(N, 64, replace=False)
        si, sj = np.meshgrid(np.arange(16), rows, indexing="ij")
        y_ref, y_seq, S = orc.gemm_samples(ref["qa"], ref["ea"], 8, ref["qw"], ref["ew"], 4, 32, si.ravel(), sj.ravel())
        got = y.cpu().numpy()[si.ravel(), sj.ravel()].astype(np.float64)
        assert (np.abs(got - y_ref) <= TOL * S + 1e-37).all()


def test_gemm_on_packed_activations_streams_too(mxb):
    """mx_gemm with already quantized tokens (M <= 16) takes the same kernel, no quantize launch."""
    dev, ref = _layer(mxb, 8, 1024, 640, seed=77, with_bias=True)
    y_ref, y_seq, S = _oracle(ref)
    a_mant = torch.from_numpy(orc.pack(ref["qa"], 8)).cuda()
    a_exp = torch.from_numpy(ref["ea"]).cuda()
    for algo in (mxb.MX_ALGO_STREAM, mxb.MX_ALGO_AUTO):
        y = mxb.mx_gemm(a_mant, a_exp, dev["fa"], dev["w_mant"], dev["w_exp"], dev["fw"], 8, 640, 1024,
                        bias=dev["bias"], algo=algo)
        err = np.abs(y.cpu().numpy().astype(np.float64) - y_ref)
        assert (err <= TOL * S + 1e-37).all()
    y_tc = mxb.mx_gemm(a_mant, a_exp, dev["fa"], dev["w_mant"], dev["w_exp"], dev["fw"], 8, 640, 1024,
                       bias=dev["bias"], algo=mxb.MX_ALGO_TCGEN05)
    assert (np.abs(y_tc.cpu().numpy().astype(np.float64) - y_ref) <= TOL * S + 1e-37).all()


def test_stream_rejects_what_it_cannot_stage(mxb):
    dev, _ = _layer(mxb, 4, 256, 64, seed=1)
    with pytest.raises(mxb.MxError):                       # block 16 weights are not streamable
        mxb.mx_linear(dev["x"], mxb.MxFormat(16, 8), dev["w_mant"], dev["w_exp"], mxb.MxFormat(16, 4), 64,
                      algo=mxb.MX_ALGO_STREAM)
    x17 = torch.zeros(17, 256, device="cuda")
    with pytest.raises(mxb.MxError):                       # more than 16 tokens
        mxb.mx_linear(x17, dev["fa"], dev["w_mant"], dev["w_exp"], dev["fw"], 64, algo=mxb.MX_ALGO_STREAM)


@pytest.mark.parametrize("T", (1, 2))
def test_rows_per_lane_kernel_over_mixed_layers(mxb, T):
    """One or two tokens, K % 512 == 0: layers of different K, width, activation and ragged N in one launch, with weight
    exponents near the top of the range and a poisoned block; enough rows that K is not cut, so the bits are the oracle's."""
    layers, refs = [], []
    for i in range(10):
        dev, ref = _layer(mxb, T, 512, 4096, seed=70 + i % 2, wa=8 - 4 * (i % 2), ww=4, with_bias=i == 3)
        if i % 2 and len(layers) > 1:
            dev["x"] = layers[1]["x"]                                   # a shared activation tensor
        layers.append(dev)
        refs.append(ref)
    for K, N, wa, ww in ((1024, 1001, 8, 3), (1536, 37, 3, 2), (512, 32, 8, 4)):
        dev, ref = _layer(mxb, T, K, N, seed=K + N, wa=wa, ww=ww, heavy=True)
        layers.append(dev)
        refs.append(ref)
    refs[-1]["ew"][3, 5], refs[-1]["ew"][9, 2] = 240, 255
    refs[-1]["qw"][9, 64:96] = 0
    layers[-1]["w_exp"].copy_(torch.from_numpy(refs[-1]["ew"]))
    layers[-1]["w_mant"].copy_(torch.from_numpy(orc.pack(refs[-1]["qw"], 4)))
    mxb.mx_linear_grouped(mxb.make_linear_args(layers))
    assert mxb.mx_poll_status() == 0
    for dev, ref in zip(layers, refs):
        _, y_seq, _ = _oracle(ref)
        y = dev["y"].cpu().numpy()
        nan = np.isnan(y_seq)
        assert np.array_equal(nan, np.isnan(y)) and np.array_equal(y[~nan], y_seq[~nan])


@pytest.mark.parametrize("T", (1, 2, 5))
def test_split_reduction_takes_every_layer_of_a_call_into_account(mxb, T):
    """K is cut over warps for few rows; the pieces must be whole stages in EVERY layer (4608 / 8 pieces is not)."""
    layers, refs = zip(*[_layer(mxb, T, K, 96, seed=K, heavy=True) for K in (4096, 4608)])
    mxb.mx_linear_grouped(mxb.make_linear_args(layers))
    assert mxb.mx_poll_status() == 0
    for dev, ref in zip(layers, refs):
        y_ref, _, S = _oracle(ref)
        assert (np.abs(dev["y"].cpu().numpy().astype(np.float64) - y_ref) <= TOL * S + 1e-37).all()


def test_two_row_and_plain_activations_of_one_call_from_two_threads(mxb):
    """Activations whose tokens pair up are quantized by launches of their own, plain ones by one launch over a table; both
    kinds and both types in one call of more layers than travel as launch parameters, issued by two threads at once."""
    import threading
    T, K, N = 2, 1024, 96
    layers, refs = [], []
    for i, (rows, dt) in enumerate(((1, torch.float32), (2, torch.float32), (1, torch.bfloat16), (2, torch.bfloat16), (1, torch.float32),
                                    (2, torch.float32))):
        x = synth.student_t_activations(T, K, 80 + i).to(dt)
        w = synth.gaussian_weights(N, K, 90 + i)
        qa, ea, _ = orc.quantize_2d(x.float().numpy(), 32, rows, 8)
        qw, ew, _ = orc.quantize(w.numpy(), 32, 4)
        refs.append(orc.gemm(qa, orc.expand_exponent_rows(ea, rows), 8, qw, ew, 4, 32))
        layers.append(dict(x=x.cuda(), fa=mxb.MxFormat(32, 8, block_rows=rows), fw=mxb.MxFormat(32, 4), N=N,
                           w_mant=torch.from_numpy(orc.pack(qw, 4)).cuda(), w_exp=torch.from_numpy(ew).cuda(),
                           y=torch.empty(T, N, device="cuda")))
    mxb.mx_linear_grouped(mxb.make_linear_args(layers))
    assert mxb.mx_poll_status() == 0
    for L, (y_ref, _, S) in zip(layers, refs):
        assert (np.abs(L["y"].cpu().numpy().astype(np.float64) - y_ref) <= TOL * S + 1e-37).all()
    results = [None, None]

    def work(t):
        stream = torch.cuda.Stream()
        mine = [dict(L, y=torch.empty_like(L["y"])) for L in layers]
        args = mxb.make_linear_args(mine)
        ws = mxb.alloc_workspace(mxb.mx_linear_grouped_workspace_bytes(args))
        stream.wait_stream(torch.cuda.default_stream())
        for _ in range(20):
            mxb.mx_linear_grouped(args, workspace=ws, stream=stream)
        stream.synchronize()
        results[t] = [L["y"] for L in mine]

    threads = [threading.Thread(target=work, args=(t,)) for t in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for ys in results:
        assert ys is not None and all(torch.equal(a, L["y"]) for a, L in zip(ys, layers))


@pytest.mark.parametrize("n_layers,shared", [(4, True), (5, True), (2, False)])
def test_a_capture_holds_only_calls_that_bring_their_tables_along(mxb, n_layers, shared):
    """Tables that travel as launch parameters can be replayed; those that are copied from the call's host memory are refused
    while a stream captures, before anything is launched."""
    devs = [_layer(mxb, 3, 512, 256, 60 + i)[0] for i in range(n_layers)]
    for d in devs:
        if shared:
            d["x"] = devs[0]["x"]
    args = mxb.make_linear_args(devs)
    ws = mxb.alloc_workspace(mxb.mx_linear_grouped_workspace_bytes(args))
    mxb.mx_linear_grouped(args, workspace=ws)
    torch.cuda.synchronize()
    want = [d["y"].clone() for d in devs]
    for d in devs:
        d["y"].zero_()
    graph = torch.cuda.CUDAGraph()
    touched = torch.zeros(1, device="cuda")
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        touched += 1
        if n_layers <= 4 and shared:
            mxb.mx_linear_grouped(args, workspace=ws)
        else:
            with pytest.raises(mxb.MxError) as e:
                mxb.mx_linear_grouped(args, workspace=ws)
            assert e.value.status == -6 and "capture" in str(e.value)
    graph.replay()
    torch.cuda.synchronize()
    assert touched.item() == 1
    for d, w in zip(devs, want):
        assert torch.equal(d["y"], w if n_layers <= 4 and shared else torch.zeros_like(w))
    mxb.mx_linear_grouped(args, workspace=ws)
    assert all(torch.equal(d["y"], w) for d, w in zip(devs, want))
    assert mxb.mx_poll_status() == 0
