"""Network parity on the GPU: calibration (formats chosen by the FL search in the forward
optimizer's order) and the integer-only forward through fxpq_net_forward, against the oracle.

The forward runs on the full batch of each workload (the launch configuration the bench times);
the oracle recomputes sampled images of that batch one by one."""
import numpy as np
import pytest
import torch

import synth
from oracle import net as onet

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def NET():
    import __graft_entry__ as g
    g.build()
    from paper_2203_12091_gb300 import net
    return net


def fmts_equal(gpu_fmts, ora_fmts):
    for nm, d in ora_fmts.items():
        if nm == "input":
            assert gpu_fmts["input"]["a"].tup() == tuple(d), nm
            continue
        for key, f in d.items():
            assert gpu_fmts[nm][key].tup() == tuple(f), (nm, key)


def _tiny():
    L = [
        {"type": "conv", "name": "c1", "C": 3, "K": 16, "R": 3, "stride": 2, "pad": 1, "relu": True, "src": None},
        {"type": "maxpool", "name": "p1", "k": 3, "stride": 2, "pad": 1},
        {"type": "conv", "name": "a", "C": 16, "K": 16, "R": 3, "stride": 1, "pad": 1, "relu": True, "src": "p1"},
        {"type": "conv", "name": "b", "C": 16, "K": 16, "R": 3, "stride": 1, "pad": 1, "relu": False, "src": "a"},
        {"type": "eltwise", "name": "e", "a": "b", "b": "p1", "relu": True},
        {"type": "avgpool", "name": "gap", "src": "e"},
        {"type": "conv", "name": "fc", "C": 16, "K": 24, "R": 1, "stride": 1, "pad": 0, "relu": False, "src": "gap"},
    ]
    plan = {"input": 7, "c1": {"w": 6, "b": 16, "a": 8}, "a": {"w": 5, "b": 16, "a": 6}, "b": {"w": 8, "b": 16, "a": 7},
            "e": {"a": 5}, "gap": {"a": 8, "r": 16}, "fc": {"w": 16, "b": 16}}
    return L, plan


def test_tiny_residual_net(NET):
    L, plan = _tiny()
    rng = np.random.default_rng(1)
    W = {}
    for l in L:
        if l["type"] == "conv":
            fan = l["C"] * l["R"] ** 2
            W[l["name"]] = ((rng.standard_normal((l["K"], l["R"], l["R"], l["C"])) * np.sqrt(2 / fan)).astype(np.float32),
                            (rng.standard_normal(l["K"]) * 0.01).astype(np.float32))
    imgs = synth.images(6, 2, hw=28)
    q = NET.build_qnet(L, W, torch.from_numpy(imgs[:4]).cuda(), plan)
    fm, qp = onet.calibrate(L, W, imgs[:4], plan)
    fmts_equal(q.fmts, fm)
    logits, s = q.forward(torch.from_numpy(imgs).cuda())
    want, ws = onet.forward(L, fm, qp, imgs)
    assert s == ws and np.array_equal(logits.cpu().numpy(), want)
    # per-layer codes of the op-by-op path agree too
    env = q.trace(torch.from_numpy(imgs).cuda())
    oenv = onet.forward_trace(L, fm, qp, imgs)
    from paper_2203_12091_gb300 import fxpq as F
    for l in L[:-1]:
        t, f = env[l["name"]]
        H, _, Cp = q.shapes[l["name"]]
        got = F.codes_to_int(t.cpu(), f, (6, H, H, Cp)).numpy()
        assert np.array_equal(got[..., : oenv[l["name"]][0].shape[-1]], oenv[l["name"]][0]), l["name"]


@pytest.mark.parametrize("R,st,pad,hw,k", [(7, 2, 3, 28, 8), (7, 2, 3, 29, 16), (3, 3, 0, 31, 6), (5, 3, 2, 28, 12), (11, 4, 2, 32, 8),
                                           (11, 4, 2, 33, 16), (3, 2, 1, 20, 2)])
def test_first_layer_from_images(NET, R, st, pad, hw, k, monkeypatch):
    """A strided first layer reads images quantized straight into its space-to-depth form, or (maps that the form does
    not cover, other paths) their codes: the same logits, and a value that is not finite is reported."""
    from paper_2203_12091_gb300 import fxpq as F
    L = [{"type": "conv", "name": "c1", "C": 3, "K": 16, "R": R, "stride": st, "pad": pad, "relu": True, "src": None},
         {"type": "avgpool", "name": "gap", "src": "c1"},
         {"type": "conv", "name": "fc", "C": 16, "K": 24, "R": 1, "stride": 1, "pad": 0, "relu": False, "src": "gap"}]
    plan = {"input": k, "c1": {"w": 8, "b": 16, "a": 8}, "gap": {"a": 8, "r": 16}, "fc": {"w": 8, "b": 16}}
    rng = np.random.default_rng(R + hw)
    W = {"c1": (rng.standard_normal((16, R, R, 3)).astype(np.float32) * 0.1, rng.standard_normal(16).astype(np.float32) * 0.01),
         "fc": (rng.standard_normal((24, 1, 1, 16)).astype(np.float32) * 0.3, rng.standard_normal(24).astype(np.float32) * 0.01)}
    imgs = synth.images(5, 2, hw=hw)
    q = NET.build_qnet(L, W, torch.from_numpy(imgs[:4]).cuda(), plan)
    fm, qp = onet.calibrate(L, W, imgs[:4], plan)
    want, ws = onet.forward(L, fm, qp, imgs)
    bad = imgs.copy()
    bad[4, 2, hw - 1, hw - 1] = np.nan
    for path in ("tc", "tc_nos2d", "simt"):
        monkeypatch.setenv("FXPQ_CONV_PATH", path)
        logits, s = q.forward(torch.from_numpy(imgs).cuda())
        assert s == ws and np.array_equal(logits.cpu().numpy(), want), path
        F.fxpq_get_device_status()
        q.forward(torch.from_numpy(bad).cuda())
        assert F.fxpq_get_device_status() == 3


def _small_net(NET):
    """A net of chained kernels of every kind, its quantized form and two batches of images with their logits."""
    L, plan = _tiny()
    rng = np.random.default_rng(12)
    W = {l["name"]: (rng.standard_normal((l["K"], l["R"], l["R"], l["C"])).astype(np.float32) * 0.2,
                     rng.standard_normal(l["K"]).astype(np.float32) * 0.01) for l in L if l["type"] == "conv"}
    imgs = [torch.from_numpy(synth.images(6, seed, hw=28)).cuda() for seed in (2, 3)]
    q = NET.build_qnet(L, W, imgs[0], plan)
    want = [q.forward(x)[0].clone() for x in imgs]
    torch.cuda.synchronize()
    assert not torch.equal(*want)
    return q, imgs, want


def test_forward_in_a_captured_graph(NET):
    """Chained launches captured as a graph: replays read the inputs of the moment."""
    from paper_2203_12091_gb300 import fxpq as F
    q, imgs, want = _small_net(NET)
    x, ws = imgs[0].clone(), F.workspace(q.workspace_bytes(6), "cuda")
    logits = torch.empty_like(want[0])
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        for _ in range(3):
            q.forward(x, logits, ws)
    for i in (1, 0, 1):
        x.copy_(imgs[i])
        logits.fill_(-1)
        graph.replay()
        assert torch.equal(logits, want[i]), i


def test_forwards_on_two_streams(NET):
    """Chained launches of two streams, each with its own workspace, interleaved."""
    from paper_2203_12091_gb300 import fxpq as F
    q, imgs, want = _small_net(NET)
    streams = [torch.cuda.Stream() for _ in range(2)]
    ws = [F.workspace(q.workspace_bytes(6), "cuda") for _ in range(2)]
    got = [[torch.empty_like(want[0]) for _ in range(20)] for _ in range(2)]
    torch.cuda.synchronize()
    for j in range(20):
        for i in range(2):
            q.forward(imgs[i], got[i][j], ws[i], streams[i])
    torch.cuda.synchronize()
    for i in range(2):
        assert all(torch.equal(g, want[i]) for g in got[i]), i


def test_smaller_workspaces(NET):
    """Scratch that holds a split reduction's shares but not the larger copies of the first layer still splits the FC layer;
    with none at all the logits are the same."""
    from paper_2203_12091_gb300 import fxpq as F
    L = [{"type": "conv", "name": "c1", "C": 3, "K": 64, "R": 7, "stride": 2, "pad": 3, "relu": True, "src": None},
         {"type": "maxpool", "name": "p1", "k": 4, "stride": 4, "pad": 0},
         {"type": "conv", "name": "fc", "C": 64, "K": 24, "R": 12, "stride": 1, "pad": 0, "relu": False, "src": "p1"}]
    plan = {"input": 8, "c1": {"w": 8, "b": 16, "a": 8}, "fc": {"w": 8, "b": 16}}
    rng = np.random.default_rng(4)
    W = {l["name"]: (rng.standard_normal((l["K"], l["R"], l["R"], l["C"])).astype(np.float32) * 0.05,
                     rng.standard_normal(l["K"]).astype(np.float32) * 0.01) for l in L if l["type"] == "conv"}
    N = 12  # 96 x 96 images: 216 row tiles, more than one round of the SMs
    imgs = torch.from_numpy(synth.images(N, 2, hw=96)).cuda()
    q = NET.build_qnet(L, W, imgs[:4], plan)
    f = q.fmts
    need = [F.fxpq_conv_workspace(F.conv_desc(N, *g, False, F.OUT_ACC64, fx, f[nm]["w"], f[nm]["b"], None))
            for nm, g, fx in (("c1", (96, 96, 3, 8, 64, 7, 7, 2, 3), f["input"]["a"]), ("fc", (12, 12, 64, 64, 24, 12, 12, 1, 0), f["c1"]["a"]))]
    full = q.workspace_bytes(N)
    slots = full - 256 - max((n + 255) // 256 * 256 for n in need)
    assert need[1] < need[0]
    out, launches = [], []
    for nbytes in (full, slots + need[1], slots):
        ws = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
        assert ws.data_ptr() % 256 == 0
        n0 = F.fxpq_launch_count()
        out.append(q.forward(imgs, ws=ws)[0].cpu())
        launches.append(F.fxpq_launch_count() - n0)
    assert torch.equal(out[0], out[1]) and torch.equal(out[0], out[2])
    assert launches[1] == launches[2] + 1, launches  # the second kernel of the split


def test_layer_dicts_without_channel_counts(NET):
    """A layer's input channels come from its weights: a trace of layers that do not state them equals one of layers that do."""
    L, plan = _tiny()
    rng = np.random.default_rng(3)
    W = {l["name"]: (rng.standard_normal((l["K"], l["R"], l["R"], l["C"])).astype(np.float32) * 0.2,
                     rng.standard_normal(l["K"]).astype(np.float32) * 0.01) for l in L if l["type"] == "conv"}
    imgs = torch.from_numpy(synth.images(3, 2, hw=28)).cuda()
    last = []
    for layers in (L, [{k: v for k, v in l.items() if k != "C"} for l in L]):
        last.append(NET.build_qnet(layers, W, imgs, plan).trace(imgs)["fc"][0].cpu())
    assert torch.equal(*last)


def test_addition_of_maps_with_different_channel_counts(NET, monkeypatch):
    """A sum of a 3-channel map (stored as 8) and an 8-channel one has 8 channels whichever comes first: the strided
    layer behind it, which the space-to-depth form reduces to its true channels, gives the same logits both ways."""
    monkeypatch.setenv("FXPQ_CONV_PATH", "tc")
    rng = np.random.default_rng(8)
    W = {nm: (rng.standard_normal(sh).astype(np.float32) * 0.2, rng.standard_normal(sh[0]).astype(np.float32) * 0.01)
         for nm, sh in (("c0", (8, 3, 3, 3)), ("c1", (16, 4, 4, 8)), ("fc", (24, 1, 1, 16)))}
    plan = {"input": 8, "c0": {"w": 8, "b": 16, "a": 8}, "e": {"a": 8}, "c1": {"w": 8, "b": 16, "a": 8}, "gap": {"a": 8, "r": 16},
            "fc": {"w": 8, "b": 16}}
    imgs = torch.from_numpy(synth.images(5, 2, hw=28)).cuda()
    out = []
    for a, b in (("p0", "c0"), ("c0", "p0")):
        L = [{"type": "maxpool", "name": "p0", "k": 3, "stride": 1, "pad": 1},
             {"type": "conv", "name": "c0", "C": 3, "K": 8, "R": 3, "stride": 1, "pad": 1, "relu": True, "src": "p0"},
             {"type": "eltwise", "name": "e", "a": a, "b": b, "relu": True},
             {"type": "conv", "name": "c1", "C": 8, "K": 16, "R": 4, "stride": 4, "pad": 0, "relu": True, "src": "e"},
             {"type": "avgpool", "name": "gap", "src": "c1"},
             {"type": "conv", "name": "fc", "C": 16, "K": 24, "R": 1, "stride": 1, "pad": 0, "relu": False, "src": "gap"}]
        q = NET.build_qnet(L, W, imgs, plan)
        logits, s = q.forward(imgs)
        out.append((logits.cpu().numpy(), s, q.fmts["c1"]["a"].tup()))
    assert np.array_equal(out[0][0], out[1][0]) and out[0][1:] == out[1][1:]


def _workload(NET, arch, batch, seed, plan_seed=None, calib=8, sample=(0, -1), pack=False):
    L = synth.ARCHS[arch]()
    W = synth.weights(arch, seed)
    plan = synth.bit_plan(arch, seed if plan_seed is None else plan_seed)
    bn = synth.bn_params(arch, seed + 100)
    imgs = synth.images(batch, seed)
    dimgs = torch.from_numpy(imgs).cuda()
    q = NET.build_qnet(L, W, dimgs[:calib], plan, bn_np=bn, pack_weights=pack)
    if pack:
        assert q.qp, "no layer took packed weights"
    fm, qp = onet.calibrate(L, W, imgs[:calib], plan, bn)
    fmts_equal(q.fmts, fm)
    logits, s = q.forward(dimgs)
    torch.cuda.synchronize()
    got = logits.cpu().numpy()
    idx = [i % batch for i in sample]
    want, ws = onet.forward(L, fm, qp, imgs[idx])
    assert s == ws
    assert np.array_equal(got[idx], want)
    from paper_2203_12091_gb300 import fxpq as F
    assert F.fxpq_get_device_status() == 0
    return got


def test_alexnet_batch256(NET):
    _workload(NET, "alexnet", 256, 5)


def test_alexnet_batch256_packed_fc_weights(NET):
    """The same workload with its three FC layers' 8-bit weights read as packed 8-bit planes
    (Sec. V-E.2) by the contraction, calibration included: formats and logits equal the oracle's."""
    _workload(NET, "alexnet", 256, 5, pack=True)


def test_resnet18_batch128(NET):
    _workload(NET, "resnet18", 128, 6)


def test_resnet18_bn_batch128(NET):
    """ResNet-18 with its BN layers kept as Scale layers (bias-free convs, aleph1 / aleph2 applied in the
    conv epilogue before ReLU), the paper's own form of the network."""
    _workload(NET, "resnet18_bn", 128, 6)


def test_bn_to_scale_bit_exact(NET):
    """fxpq_bn_to_scale against the oracle's fp32 formula, bit for bit (every step correctly rounded)."""
    from oracle import bn_to_scale
    from paper_2203_12091_gb300 import fxpq as F
    rng = np.random.default_rng(31)
    n = 10007
    g = rng.uniform(-2, 2, n).astype(np.float32)
    b = rng.normal(0, 1, n).astype(np.float32)
    mu = rng.normal(0, 3, n).astype(np.float32)
    var = np.concatenate([rng.uniform(0, 5, n - 3), [0.0, 1e-30, 1e6]]).astype(np.float32)
    d = [torch.from_numpy(t).cuda() for t in (g, b, mu, var)]
    a1 = torch.empty(n, dtype=torch.float32, device="cuda")
    a2 = torch.empty(n, dtype=torch.float32, device="cuda")
    F.fxpq_bn_to_scale(*d, NET.BN_EPS, a1, a2)
    w1, w2 = bn_to_scale(g, b, mu, var, NET.BN_EPS)
    assert np.array_equal(a1.cpu().numpy().view(np.uint32), w1.view(np.uint32))
    assert np.array_equal(a2.cpu().numpy().view(np.uint32), w2.view(np.uint32))


@pytest.mark.parametrize("plan_seed", [7, 38])
def test_vgg16_batch64_plans(NET, plan_seed):
    _workload(NET, "vgg16", 64, 7, plan_seed=plan_seed, sample=(0,))


def test_vgg16_batch64_packed_fc_weights(NET):
    """VGG-16 with fc6 / fc7 reading packed weights (4..8 bits per the plan; fc8's are 16-bit and stay
    fp16 code planes)."""
    _workload(NET, "vgg16", 64, 7, plan_seed=7, sample=(0,), pack=True)


def test_single_conv_workload_end_to_end(NET):
    """The single-conv workload (batch 8, 64 -> 64 channels, 32 x 32 maps, 3 x 3, stride 1, pad 1): He-normal
    weights, ReLU(N(0,1)) inputs, N(0, 0.01) biases, 8-bit weights and activations with FL searched over
    0..15 (16-bit bias), the output requantized to 8 bits with its FL searched on the exact C-Block output.
    Every format and every code equals the oracle's."""
    import oracle
    from paper_2203_12091_gb300 import fxpq as F
    N, H, C, K = 8, 32, 64, 64
    g = torch.Generator().manual_seed(91)
    x = torch.relu(torch.randn(N, H, H, C, generator=g)).numpy()
    w = (torch.randn(K, 3, 3, C, generator=g) * np.sqrt(2.0 / (9 * C))).numpy().astype(np.float32)
    b = (torch.randn(K, generator=g) * 0.01).numpy().astype(np.float32)
    fmt_gpu, fmt_ora = {}, {}
    for nm, t, k in (("x", x, 8), ("w", w, 8), ("b", b, 16)):
        err, best, st = F.fl_search(torch.from_numpy(t).cuda().reshape(-1), -1, k, k, 0, 15)
        S = F.stats_from_device(st).is_signed
        fmt_gpu[nm] = F.fmt(k, S, int(best.cpu()[0]))
        _, obest, oS, _ = oracle.fl_search(t.reshape(-1), -1, k, k, 0, 15)
        fmt_ora[nm] = (k, oS, int(obest[0]))
        assert fmt_gpu[nm].tup() == fmt_ora[nm], nm
    xq = torch.empty(N * H * H * C, dtype=torch.float16, device="cuda")
    F.fxpq_quantize_rows(torch.from_numpy(x).cuda(), N * H * H, C, fmt_gpu["x"], C, xq)
    wq = torch.empty(K * 9 * C, dtype=torch.float16, device="cuda")
    F.fxpq_quantize_rows(torch.from_numpy(w).cuda(), K * 9, C, fmt_gpu["w"], C, wq)
    bq = torch.empty(K, dtype=torch.int32, device="cuda")
    F.fxpq_quantize(torch.from_numpy(b).cuda(), fmt_gpu["b"], F.DT_I32, bq)
    # the exact C-Block output's fp32 image, its FL search, then the codes
    f32 = torch.empty(N * H * H * K, dtype=torch.float32, device="cuda")
    d = F.conv_desc(N, H, H, C, C, K, 3, 3, 1, 1, True, F.OUT_F32, fmt_gpu["x"], fmt_gpu["w"], fmt_gpu["b"], None)
    F.fxpq_conv_fwd(d, xq, wq, bq, f32)
    _, ybest, yst = F.fl_search(f32, -1, 8, 8, 0, 15)
    fy = F.fmt(8, F.stats_from_device(yst).is_signed, int(ybest.cpu()[0]))
    y = torch.empty(N * H * H * K, dtype=torch.float16, device="cuda")
    d = F.conv_desc(N, H, H, C, C, K, 3, 3, 1, 1, True, F.OUT_CODES, fmt_gpu["x"], fmt_gpu["w"], fmt_gpu["b"], fy)
    F.fxpq_conv_fwd(d, xq, wq, bq, y)
    torch.cuda.synchronize()
    qx = oracle.quantize(x, *fmt_ora["x"]).reshape(x.shape)
    qw = oracle.quantize(w, *fmt_ora["w"]).reshape(w.shape)
    qb = oracle.quantize(b, *fmt_ora["b"])
    v, s = oracle.cblock(oracle.conv2d(qx, qw, 1, 1), fmt_ora["x"][2] + fmt_ora["w"][2], qb, fmt_ora["b"][2], True)
    assert np.array_equal(f32.cpu().numpy().reshape(v.shape), oracle.to_f32(v, s))
    _, oyb, oyS, _ = oracle.fl_search(oracle.to_f32(v, s).reshape(-1), -1, 8, 8, 0, 15)
    assert fy.tup() == (8, oyS, int(oyb[0]))
    want = oracle.requant(v, s, 8, oyS, int(oyb[0]))
    assert np.array_equal(F.codes_to_int(y.cpu(), fy, (N, H, H, K)).numpy(), want)
