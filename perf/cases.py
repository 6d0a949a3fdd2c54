"""The measured cases: what programs ask of this library, through its public
entry points, over the sizes, types and options that they use.

Families (the `family` of a case):

  matmul    nk_matmul: FP32 operands at every precision, or operands the
            caller keeps in BF16 (activations and weights of a served layer)
  grouped   one persistent launch of a plan of uneven BF16 GEMMs
  conv      nk_conv2d_nhwc_hwcf: FP32, BF16 with packed weights, E4M3
  nchw      nk_conv2d_nchw_fchw: the few-channel image convolution
  forward   forward.ResNetStack, captured in a CUDA graph as a server would
  train     a mini-batch step of the tile-cost model (gradient, then Adam)

Schedules are the built-in ones, and buffers (outputs, workspaces, packed
weights, plans) are kept by the caller, as a program with a loop keeps them.
"""
import math

import torch

from paper_2307_16080_gb300 import forward, nk
from paper_2307_16080_gb300 import nk_tune as nt


def listed():
    return [
        # a small FP32 product on its own: launch and latency
        dict(name="matmul_f32_256", family="matmul", prec="f32", M=256, N=256, K=256, bias=False, relu=False, ew="",
             b_t=False, cast=False),
        # a plain FP32 layer whose extents nobody rounded: odd leading dimensions
        dict(name="matmul_f32_odd", family="matmul", prec="f32", M=1531, N=2047, K=1021, bias=True, relu=True, ew="",
             b_t=False, cast=False),
        # the up-projection of an MLP block: activations and weights [out, in]
        # held in BF16, bias and GELU fused
        dict(name="linear_bf16_gelu", family="matmul", prec="bf16", M=4096, N=4096, K=1024, bias=True, relu=False,
             ew="gelu", b_t=True, cast=True),
        # the precision sweep's large product: FP32 operands, BF16 tensor cores
        dict(name="matmul_bf16_8192", family="matmul", prec="bf16", M=8192, N=8192, K=8192, bias=False, relu=False,
             ew="", b_t=False, cast=False),
        # the sweep's 4096 product in E4M3: amax, quantisation and product per call
        dict(name="matmul_fp8_4096", family="matmul", prec="fp8", M=4096, N=4096, K=4096, bias=False, relu=False,
             ew="", b_t=False, cast=False),
        # FP32 accuracy on the tensor cores, ragged extents, a Linear layer's epilogue
        dict(name="matmul_bf16x3_ragged", family="matmul", prec="bf16x3", M=3001, N=2002, K=1999, bias=True,
             relu=True, ew="", b_t=False, cast=False),
        # the grouped workload: 512 uneven GEMMs in one launch
        dict(name="grouped_512", family="grouped", G=512, lo=32, hi=2048),
        # the FP32 convolution block (bias + ReLU)
        dict(name="conv_f32_8x56x56x64", family="conv", prec="f32", n=8, h=56, w=56, c=64, f=64, k=3, stride=1,
             out_bf16=False),
        # the same layer of a training- or serving-sized batch in BF16, feeding the next layer
        dict(name="conv_bf16_128x56x56x64", family="conv", prec="bf16", n=128, h=56, w=56, c=64, f=64, k=3, stride=1,
             out_bf16=True),
        # the tuning experiment's image convolution over a batch of images
        dict(name="nchw_16x1280x1280", family="nchw", n=16, ci=1, h=1280, w=1280, co=3, k=3),
        # the 20 layers feeding each other, at the middle batch
        dict(name="forward_batch8", family="forward", batch=8),
        # one step of the cost model's training at its own mini-batch
        dict(name="train_1024", family="train", batch=1024),
    ]


def _log(rng, lo, hi, multiple=1):
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return max(multiple, int(round(v / multiple)) * multiple)


def draw(rng):
    fam = rng.choice(["matmul"] * 5 + ["grouped", "conv", "conv", "conv", "nchw", "forward", "train"])
    if fam == "matmul":
        prec = rng.choice(["f32", "bf16", "bf16", "fp8", "bf16x3"])
        cast = prec == "bf16" and rng.random() < 0.5
        hi = {"f32": 2048, "bf16": 8192, "fp8": 8192, "bf16x3": 4096}[prec]
        lo = 64 if prec == "f32" else 128
        mult = rng.choice([1, 8, 64])
        return dict(family="matmul", prec=prec, M=_log(rng, lo, hi, mult), N=_log(rng, lo, hi, mult),
                    K=_log(rng, lo, hi, 8 if cast else mult), bias=rng.random() < 0.5, relu=rng.random() < 0.3,
                    ew=rng.choice(["", "", "gelu", "silu"]) if cast else "", b_t=cast or rng.random() < 0.3, cast=cast)
    if fam == "grouped":
        return dict(family="grouped", G=_log(rng, 16, 512), lo=32, hi=rng.choice([512, 1024, 2048]))
    if fam == "conv":
        prec = rng.choice(["f32", "bf16", "bf16", "bf16", "fp8"])
        h, c = rng.choice([(56, 64), (28, 128), (14, 256), (7, 512), (rng.randint(9, 60), 8 * rng.randint(4, 32))])
        f = c if rng.random() < 0.6 else min(2 * c, 512)
        w = h if rng.random() < 0.7 else h + rng.randint(1, 5)
        k, stride = rng.choice([1, 3, 3, 3]), rng.choice([1, 1, 2])
        most = (1e10 if prec == "f32" else 2e11) / (2.0 * h * w * c * f * k * k / stride ** 2)   # images
        return dict(family="conv", prec=prec, n=_log(rng, 1, max(1.0, min(most, 16 if prec == "f32" else 128))), h=h,
                    w=w, c=c, f=f, k=k, stride=stride, out_bf16=prec == "bf16" and rng.random() < 0.7)
    if fam == "nchw":
        return dict(family="nchw", n=_log(rng, 1, 16), ci=rng.choice([1, 1, 3]), h=rng.randint(240, 1280),
                    w=rng.randint(240, 1280), co=rng.choice([1, 3, 4]), k=rng.choice([1, 3, 3, 5]))
    if fam == "forward":
        return dict(family="forward", batch=_log(rng, 1, 32))
    return dict(family="train", batch=_log(rng, 64, 4096))


# ------------------------------------------------------------------ inputs
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _normal(g, *shape, sigma=1.0):
    return torch.randn(*shape, generator=g, device="cuda") * sigma


def _outliers(g, *shape):
    """N(0,1) with one entry in a hundred scaled by 100."""
    x = torch.randn(*shape, generator=g, device="cuda")
    return torch.where(torch.rand(*shape, generator=g, device="cuda") < 0.01, x * 100.0, x)


def _uniform(g, *shape, lo=-1.0, hi=1.0):
    return torch.rand(*shape, generator=g, device="cuda") * (hi - lo) + lo


def _matmul_inputs(case, seed):
    g = _gen(seed)
    M, N, K = case["M"], case["N"], case["K"]
    if case["cast"]:
        # a layer's activations and He-scaled weights, both kept in BF16
        A = _normal(g, M, K).bfloat16()
        B = _normal(g, N, K, sigma=math.sqrt(2.0 / K)).bfloat16().t()
    elif case["prec"] == "f32":
        A, B = _uniform(g, M, K), _uniform(g, N, K).t() if case["b_t"] else _uniform(g, K, N)
    else:
        A, B = _outliers(g, M, K), _outliers(g, N, K).t() if case["b_t"] else _outliers(g, K, N)
    return A, B, _uniform(g, N, lo=-0.1, hi=0.1) if case["bias"] else None


def _group_shapes(case):
    """(M, N, K) of the groups, log-uniform in multiples of 16: a plan's sizes
    are part of the program, so they do not depend on the seed."""
    u = torch.rand(case["G"], 3, generator=torch.Generator().manual_seed(4), dtype=torch.float64)
    lo, hi = case["lo"], case["hi"]
    x = torch.exp(math.log(lo) + (math.log(hi) - math.log(lo)) * u)
    return ((x / 16).round().clamp(lo // 16, hi // 16).long() * 16).tolist()


def _grouped_inputs(case, seed):
    g = _gen(seed)
    shapes = _group_shapes(case)
    As = [_uniform(g, M, K).bfloat16() for M, _, K in shapes]
    Bts = [_uniform(g, N, K).bfloat16() for _, N, K in shapes]
    return shapes, As, Bts


def _conv_out(case):
    pad = case["k"] // 2
    return pad, (case["h"] + 2 * pad - case["k"]) // case["stride"] + 1, (case["w"] + 2 * pad - case["k"]) // case["stride"] + 1


def _conv_inputs(case, seed):
    g = _gen(seed)
    k, c, f = case["k"], case["c"], case["f"]
    I = _normal(g, case["n"], case["h"], case["w"], c).abs_()
    W = _normal(g, k, k, c, f, sigma=math.sqrt(2.0 / (k * k * c)))
    return I.bfloat16() if case["prec"] == "bf16" else I, W, _uniform(g, f, lo=-0.1, hi=0.1)


def _nchw_inputs(case, seed):
    g = _gen(seed)
    return (_uniform(g, case["n"], case["ci"], case["h"], case["w"]),
            _normal(g, case["co"], case["ci"], case["k"], case["k"], sigma=math.sqrt(2.0 / (case["ci"] * case["k"] ** 2))),
            _uniform(g, case["co"], lo=-0.1, hi=0.1))


def _train_inputs(case, seed):
    g = _gen(seed)
    s0, s1 = 1.0 / math.sqrt(16.0), 1.0 / math.sqrt(128.0)
    P = torch.cat([_normal(g, 128 * 16, sigma=s0), _normal(g, 128, sigma=0.1), _normal(g, 128 * 128, sigma=s1),
                   _normal(g, 128, sigma=0.1), _normal(g, 128, sigma=s1), _normal(g, 1, sigma=0.1)])
    X = _uniform(g, case["batch"], 16, lo=0.0, hi=1.0)
    t = _normal(g, case["batch"])
    # moments of a run that is under way
    m, v = _normal(g, P.numel(), sigma=1e-3), _uniform(g, P.numel(), lo=1e-6, hi=1e-4)
    return P, X, t, m, v


_STEP, _LR = 500, 1e-3


# ------------------------------------------------------------------ the calls
def prepare(case, seed):
    fam = case["family"]
    if fam == "matmul":
        A, B, bias = _matmul_inputs(case, seed)
        C = torch.empty(case["M"], case["N"], device="cuda")
        ws = nk.workspace(nk.nk_matmul_workspace_size(A, B, C, case["prec"]), C.device)
        return dict(case=case, A=A, B=B, bias=bias, C=C, ws=ws, ew=[(case["ew"],)] if case["ew"] else None)
    if fam == "grouped":
        shapes, As, Bts = _grouped_inputs(case, seed)
        flat = torch.empty(sum(M * N for M, N, _ in shapes), device="cuda")
        Cs, at = [], 0
        for M, N, _ in shapes:
            Cs.append(flat[at:at + M * N].view(M, N))
            at += M * N
        groups, G = nk.make_groups(As, Bts, Cs)
        return dict(case=case, keep=(As, Bts, Cs, groups), C=flat, plan=_Plan(nk.nk_grouped_plan_create(groups, G)))
    if fam == "conv":
        I, W, bias = _conv_inputs(case, seed)
        pad, oh, ow = _conv_out(case)
        O = torch.empty(case["n"], oh, ow, case["f"], device="cuda",
                        dtype=torch.bfloat16 if case["out_bf16"] else torch.float32)
        if case["prec"] == "bf16":
            W = nk.nk_conv2d_pack_weights(W)
        st, pd = (case["stride"],) * 2, (pad,) * 4
        ws = nk.workspace(nk.nk_conv2d_workspace_size(I, W, O, st, (1, 1), pd, case["prec"]), O.device)
        return dict(case=case, I=I, W=W, bias=bias, O=O, stride=st, pad=pd, ws=ws)
    if fam == "nchw":
        I, K, bias = _nchw_inputs(case, seed)
        O = torch.empty(case["n"], case["co"], case["h"] - case["k"] + 1, case["w"] - case["k"] + 1, device="cuda")
        return dict(case=case, I=I, K=K, bias=bias, O=O)
    if fam == "forward":
        net = forward.ResNetStack(case["batch"], "cuda", seed=int(seed))
        net.bind(_uniform(_gen(seed), case["batch"], 56, 56, 64, lo=0.0).bfloat16())
        net.run()   # loads the kernels before the capture
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            net.run()
        return dict(case=case, net=net, graph=graph)
    P, X, t, m, v = _train_inputs(case, seed)
    ws = torch.empty(nt.nk_mlp_workspace_size(case["batch"]), dtype=torch.uint8, device="cuda")
    return dict(case=case, P=P, X=X, t=t, m=m, v=v, g=torch.empty_like(P), loss=torch.empty(1, device="cuda"), ws=ws,
                step=_STEP)


class _Plan:
    """Owns a grouped plan: its device table is freed with the state."""

    def __init__(self, handle):
        self.handle = handle

    def __del__(self):
        nk.nk_grouped_plan_destroy(self.handle)


def run(state):
    case, s = state["case"], state
    fam = case["family"]
    if fam == "matmul":
        return nk.nk_matmul(s["A"], s["B"], s["C"], case["prec"], bias=s["bias"], relu=case["relu"], ws=s["ws"],
                            ew=s["ew"])
    if fam == "grouped":
        nk.nk_grouped_plan_run(s["plan"].handle)
        return s["C"]
    if fam == "conv":
        return nk.nk_conv2d_nhwc_hwcf(s["I"], s["W"], s["O"], s["stride"], (1, 1), s["pad"], case["prec"],
                                      bias=s["bias"], relu=True, ws=s["ws"])
    if fam == "nchw":
        return nk.nk_conv2d_nchw_fchw(s["I"], s["K"], s["O"], bias=s["bias"])
    if fam == "forward":
        s["graph"].replay()
        return s["net"].outputs[-1]
    nt.nk_mlp_grad(s["P"], s["X"], s["t"], s["g"], s["loss"], s["ws"])
    nt.nk_mlp_adam(s["P"], s["g"], s["m"], s["v"], s["step"], lr=_LR)
    s["step"] += 1
    return dict(loss=s["loss"], grad=s["g"], params=s["P"])


# ------------------------------------------------------------------ the work
def work(case):
    fam = case["family"]
    if fam == "matmul":
        M, N, K = case["M"], case["N"], case["K"]
        return dict(bytes=(2 if case["cast"] else 4) * (M * K + K * N) + 4 * M * N, flops=2.0 * M * N * K)
    if fam == "grouped":
        shapes = _group_shapes(case)
        return dict(bytes=sum(2 * (M * K + K * N) + 4 * M * N for M, N, K in shapes),
                    flops=sum(2.0 * M * N * K for M, N, K in shapes))
    if fam == "conv":
        _, oh, ow = _conv_out(case)
        c, f, taps = case["c"], case["f"], case["k"] ** 2
        in_size, out_size = (2 if case["prec"] == "bf16" else 4), (2 if case["out_bf16"] else 4)
        return dict(bytes=in_size * (case["n"] * case["h"] * case["w"] * c + taps * c * f) + out_size * case["n"] * oh * ow * f,
                    flops=2.0 * case["n"] * oh * ow * f * taps * c)
    if fam == "nchw":
        oh, ow = case["h"] - case["k"] + 1, case["w"] - case["k"] + 1
        return dict(bytes=4 * case["n"] * (case["ci"] * case["h"] * case["w"] + case["co"] * oh * ow),
                    flops=2.0 * case["n"] * case["co"] * oh * ow * case["ci"] * case["k"] ** 2)
    if fam == "forward":
        flops, weights = 0.0, 0
        for L in _layers():
            weights += L["k"] ** 2 * L["c"] * L["f"]
            flops += 2.0 * case["batch"] * L["oh"] ** 2 * L["f"] * L["k"] ** 2 * L["c"]
        return dict(bytes=2 * weights + case["batch"] * (2 * 56 * 56 * 64 + 4 * 7 * 7 * 512), flops=flops)
    n = 128 * 16 + 128 + 128 * 128 + 128 + 128 + 1
    return dict(bytes=4 * (8 * n + 17 * case["batch"]), flops=6.0 * case["batch"] * (128 * 16 + 128 * 128 + 128))


def _layers():
    """The stack's layers in order (kernel, stride, channels, output extent)."""
    out = [dict(k=3, s=1, c=64, f=64, oh=56)] * 4
    cin = 64
    for f, oh in ((128, 28), (256, 14), (512, 7)):
        out = out + [dict(k=3, s=2, c=cin, f=f, oh=oh), dict(k=1, s=2, c=cin, f=f, oh=oh)]
        out = out + [dict(k=3, s=1, c=f, f=f, oh=oh)] * 3
        cin = f
    return out + [dict(k=1, s=1, c=512, f=512, oh=7)]


# ------------------------------------------------------------------ 64 bits
def _conv64(I, W, stride, pad):
    """NHWC x HWCF in 64 bits, one matrix product per filter tap."""
    n, h, w, c = I.shape
    kh, kw, _, f = W.shape
    oh, ow = (h + 2 * pad - kh) // stride + 1, (w + 2 * pad - kw) // stride + 1
    x = torch.zeros(n, h + 2 * pad, w + 2 * pad, c, dtype=torch.float64, device=I.device)
    x[:, pad:pad + h, pad:pad + w] = I.double()
    out = torch.zeros(n * oh * ow, f, dtype=torch.float64, device=I.device)
    for a in range(kh):
        for b in range(kw):
            v = x[:, a:a + (oh - 1) * stride + 1:stride, b:b + (ow - 1) * stride + 1:stride]
            out += v.reshape(n * oh * ow, c) @ W[a, b].double()
    return out.view(n, oh, ow, f)


def _erf_gelu(z):
    return 0.5 * z * torch.erfc(-z / math.sqrt(2.0))


def exact(case, seed):
    fam = case["family"]
    if fam == "matmul":
        A, B, bias = _matmul_inputs(case, seed)
        C = A.double() @ B.double()
        if bias is not None:
            C += bias.double()
        if case["relu"]:
            C = C.clamp_(min=0.0)
        if case["ew"] == "gelu":
            C = _erf_gelu(C)
        elif case["ew"] == "silu":
            C = C * torch.sigmoid(C)
        return C
    if fam == "grouped":
        _, As, Bts = _grouped_inputs(case, seed)
        return torch.cat([(a.double() @ b.double().t()).reshape(-1) for a, b in zip(As, Bts)])
    if fam == "conv":
        I, W, bias = _conv_inputs(case, seed)
        pad, _, _ = _conv_out(case)
        return (_conv64(I, W, case["stride"], pad) + bias.double()).clamp_(min=0.0)
    if fam == "nchw":
        I, K, bias = _nchw_inputs(case, seed)
        oh, ow = case["h"] - case["k"] + 1, case["w"] - case["k"] + 1
        O = bias.double().view(1, -1, 1, 1).repeat(case["n"], 1, oh, ow)
        for co in range(case["co"]):
            for ci in range(case["ci"]):
                for a in range(case["k"]):
                    for b in range(case["k"]):
                        O[:, co] += I[:, ci, a:a + oh, b:b + ow].double() * K[co, ci, a, b].double()
        return O
    if fam == "forward":
        net = forward.ResNetStack(case["batch"], "cuda", seed=int(seed))   # only for the weights it draws
        W = [torch.from_numpy(w).cuda() for w in net.weights32]
        b = [torch.from_numpy(v).cuda().double() for v in net.bias32]
        x = _uniform(_gen(seed), case["batch"], 56, 56, 64, lo=0.0).bfloat16().double()
        conv = lambda v, i, s, p: _conv64(v, W[i], s, p) + b[i]  # noqa: E731
        for i in range(4):
            x = conv(x, i, 1, 1).clamp_(min=0.0)
        for i in (4, 9, 14):
            a, p = conv(x, i, 2, 1).clamp_(min=0.0), conv(x, i + 1, 2, 0)
            a = conv(conv(a, i + 2, 1, 1).clamp_(min=0.0), i + 3, 1, 1).clamp_(min=0.0)
            x = (conv(a, i + 4, 1, 1) + p).clamp_(min=0.0)
        return conv(x, 19, 1, 0).clamp_(min=0.0)
    P, X, t, m, v = (q.double() for q in _train_inputs(case, seed))
    P.requires_grad_(True)
    W1, b1, W2, b2, W3, b3 = P.split([128 * 16, 128, 128 * 128, 128, 128, 1])
    h1 = _erf_gelu(X @ W1.view(128, 16).t() + b1)
    h2 = _erf_gelu(h1 @ W2.view(128, 128).t() + b2)
    loss = ((h2 @ W3 + b3 - t) ** 2).mean()
    loss.backward()
    g = P.grad
    m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
    mh, vh = m / (1 - 0.9 ** _STEP), v / (1 - 0.999 ** _STEP)
    return dict(loss=loss.detach().view(1), grad=g, params=P.detach() - _LR * mh / (vh.sqrt() + 1e-8))
