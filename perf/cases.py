"""The work a user of this library has it do, as measurable cases.

A training loop that keeps activations in Tucker form calls the library once per trained layer and step in each
direction: compress in the forward pass, the weight gradient in the backward pass.  One pass of a case is such a
layer-step (kinds "conv" and "linear", through LayerRunner), the layer-steps of one training step together (kind
"step", through StepRunner), the cold start of a layer (kind "cold"), or a layer-step whose tensors live in host
memory (kind "host").

Inputs have the structure the method is made for: a Tucker tensor whose energy falls off geometrically along every
mode, plus a little noise, with previous factors one small rotation away; output gradients are Gaussian.
"""
import math

import torch

from paper_2505_05086_b200.runner import LayerRunner, StepRunner

# Trained layers of the benchmark's fine-tuning workloads: conv (C, H, cout, k, stride, pad, groups, ranks) with
# ranks at the energy threshold the benchmark uses; linear (N, Din, Dout, ranks).
STEPS = {
    "resnet18-last4": ("conv", [
        (256, 14, 512, 3, 2, 1, 1, (3, 3, 3, 4)), (512, 7, 512, 3, 1, 1, 1, (4, 4, 4, 4)),
        (512, 7, 512, 3, 1, 1, 1, (3, 4, 4, 3)), (512, 7, 512, 3, 1, 1, 1, (4, 4, 4, 3))]),
    "mobilenetv2-last5": ("conv", [
        (960, 7, 160, 1, 1, 0, 1, (2, 3, 2, 3)), (160, 7, 960, 1, 1, 0, 1, (4, 4, 3, 3)),
        (960, 7, 960, 3, 1, 1, 960, (3, 4, 3, 3)), (960, 7, 320, 1, 1, 0, 1, (3, 4, 2, 3)),
        (320, 7, 1280, 1, 1, 0, 1, (4, 4, 3, 3))]),
    "resnet34-sweep": ("conv", [
        (64, 56, 64, 3, 1, 1, 1, (3, 4, 4, 4)), (64, 56, 128, 3, 2, 1, 1, (4, 4, 4, 4)),
        (64, 56, 128, 1, 2, 0, 1, (3, 3, 4, 3)), (128, 28, 128, 3, 1, 1, 1, (3, 3, 3, 3)),
        (128, 28, 256, 3, 2, 1, 1, (3, 3, 4, 4)), (128, 28, 256, 1, 2, 0, 1, (4, 4, 3, 3)),
        (256, 14, 256, 3, 1, 1, 1, (3, 4, 3, 4)), (256, 14, 512, 3, 2, 1, 1, (4, 3, 3, 4)),
        (256, 14, 512, 1, 2, 0, 1, (4, 4, 4, 4)), (512, 7, 512, 3, 1, 1, 1, (3, 3, 3, 3))]),
    "vit-base-mlp": ("linear", [(197, 768, 3072, (8, 32, 64)), (197, 3072, 768, (8, 32, 64))]),
    "llm-tokens": ("linear", [
        (512, 2048, 2048, (8, 20, 20)), (512, 2048, 5632, (8, 20, 20)), (512, 5632, 2048, (8, 20, 20))]),
}
MOST = 128 * 64 * 56 * 56        # elements of the largest activation of a single-layer case


def listed():
    return [
        # one 3x3 conv on a tiny batch: nothing but launches and latency
        dict(name="conv-small", kind="conv", B=8, C=32, H=16, W=16, cout=32, k=3, stride=1, pad=1, groups=1,
             r1=4, r2=8, r3=8, r4=8, bf16=False),
        # fine-tuning the last layers of an image classifier: 14x14 and 7x7 maps, the layers of a step together
        dict(name="step-resnet18-last4", kind="step", layers="resnet18-last4", B=64, N=0, more=0, bf16=False),
        dict(name="step-mobilenetv2-last5", kind="step", layers="mobilenetv2-last5", B=128, N=0, more=0, bf16=False),
        # every conv shape of a deeper one, 56x56 down to 7x7: the benchmark's headline and the largest case
        dict(name="step-resnet34-sweep", kind="step", layers="resnet34-sweep", B=128, N=0, more=0, bf16=False),
        # a middle layer under mixed precision
        dict(name="conv-28-bf16", kind="conv", B=128, C=128, H=28, W=28, cout=128, k=3, stride=1, pad=1, groups=1,
             r1=3, r2=3, r3=3, r4=3, bf16=True),
        # another input resolution and a last, short batch: nothing a multiple of anything, ranks above four
        dict(name="conv-ragged", kind="conv", B=50, C=116, H=27, W=27, cout=90, k=3, stride=2, pad=1, groups=1,
             r1=5, r2=6, r3=5, r4=5, bf16=False),
        # the MLP of a vision transformer block and the projections of a language model block, bf16 tokens
        dict(name="step-vit-mlp", kind="step", layers="vit-base-mlp", B=32, N=197, more=0, bf16=True),
        dict(name="step-llm-tokens", kind="step", layers="llm-tokens", B=8, N=512, more=0, bf16=True),
        # a token layer trained in fp32
        dict(name="linear-tokens-f32", kind="linear", B=16, N=197, D=768, cout=768, r1=8, r2=16, r3=32, bf16=False),
        # a classifier head: two modes, no token dimension
        dict(name="linear-head", kind="linear", B=128, N=0, D=1280, cout=1000, r1=16, r2=0, r3=16, bf16=False),
        # the first step of a layer: factors from Gaussian test matrices the library draws itself
        dict(name="cold-start", kind="cold", B=64, C=128, H=28, W=28, cout=128, k=3, stride=1, pad=1, groups=1,
             r1=4, r2=4, r3=4, r4=4, bf16=False),
        # tensors offloaded to (pinned) host memory: the whole layer-step from there and back
        dict(name="host-step", kind="host", B=64, C=128, H=28, W=28, cout=128, k=3, stride=1, pad=1, groups=1,
             r1=3, r2=3, r3=3, r4=3, bf16=False),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_conv(rng, kind, most):
    H = rng.choice((7, 14, 16, 28, 56)) if rng.random() < 0.5 else _log(rng, 6, 56)
    W = H if rng.random() < 0.75 else _log(rng, 6, 56)
    C = _log(rng, 16, 512)
    B = min(_log(rng, 4, 128), max(2, most // (C * H * W)))
    B = B // 8 * 8 if B >= 8 and rng.random() < 0.5 else B
    k, groups, cout = rng.choice((1, 3, 3, 5)), 1, _log(rng, 16, 512)
    if rng.random() < 0.2:
        cout, groups = C, C
    cout = min(cout, max(2, most // (B * H * W))) if groups == 1 else cout
    r = [min(rng.randint(2, 5) if rng.random() < 0.7 else rng.randint(5, 8), d) for d in (B, C, H, W)]
    return dict(kind=kind, B=B, C=C, H=H, W=W, cout=cout, k=k, stride=rng.choice((1, 1, 2)), pad=k // 2,
                groups=groups, r1=r[0], r2=r[1], r3=r[2], r4=r[3], bf16=rng.random() < 0.3)


def draw(rng):
    what = rng.choice(("conv", "conv", "conv", "step-conv", "step-conv", "tokens", "tokens", "step-tokens", "head",
                       "cold", "host"))
    if what in ("conv", "cold", "host"):
        return _draw_conv(rng, what, MOST if what == "conv" else MOST // 4)
    if what == "step-conv":
        layers = rng.choice(("resnet18-last4", "mobilenetv2-last5", "resnet34-sweep"))
        return dict(kind="step", layers=layers, B=_log(rng, 8, 128), N=0, more=rng.randint(0, 1),
                    bf16=rng.random() < 0.3)
    if what == "step-tokens":
        layers = rng.choice(("vit-base-mlp", "llm-tokens"))
        lo, hi = (49, 256) if layers == "vit-base-mlp" else (64, 512)
        return dict(kind="step", layers=layers, B=_log(rng, 8, 32 if layers == "vit-base-mlp" else 8),
                    N=_log(rng, lo, hi), more=0, bf16=rng.random() < 0.75)
    if what == "head":
        B, D, cout = _log(rng, 32, 512), _log(rng, 128, 4096), _log(rng, 10, 2000)
        r = rng.randint(4, 24)                        # a matrix has one rank
        return dict(kind="linear", B=B, N=0, D=D, cout=cout, r1=r, r2=0, r3=r, bf16=rng.random() < 0.3)
    B, N, D, cout = _log(rng, 4, 32), _log(rng, 32, 512), _log(rng, 128, 3072), _log(rng, 128, 3072)
    if rng.random() < 0.5:
        D, cout = (D + 63) // 64 * 64, (cout + 63) // 64 * 64
    B = max(4, min(B, MOST // 2 // (N * max(D, cout))))
    r1, r2 = min(B, rng.randint(4, 8)), 4 * rng.randint(3, 8)
    return dict(kind="linear", B=B, N=N, D=D, cout=cout, r1=r1, r2=r2, r3=4 * rng.randint(2, min(16, r1 * r2 // 12)),
                bf16=rng.random() < 0.5)


def layers_of(case):
    """The case's layers: keyword arguments of LayerRunner."""
    c = case
    if c["kind"] in ("conv", "cold", "host"):
        return [dict(kind="conv", dims=(c["B"], c["C"], c["H"], c["W"]), ranks=(c["r1"], c["r2"], c["r3"], c["r4"]),
                     cout=c["cout"], k=c["k"], stride=c["stride"], pad=c["pad"], groups=c["groups"], bf16=c["bf16"])]
    if c["kind"] == "linear":
        d = (c["B"], c["N"], c["D"]) if c["N"] else (c["B"], c["D"])
        r = (c["r1"], c["r2"], c["r3"]) if c["N"] else (c["r1"], c["r3"])
        return [dict(kind="linear", dims=d, ranks=r, cout=c["cout"], bf16=c["bf16"])]
    kind, rows = STEPS[c["layers"]]
    if kind == "conv":
        return [dict(kind="conv", dims=(c["B"], C, H, H), ranks=tuple(x + c["more"] for x in r), cout=cout, k=k,
                     stride=s, pad=p, groups=g, bf16=c["bf16"]) for C, H, cout, k, s, p, g, r in rows]
    return [dict(kind="linear", dims=(c["B"], c["N"], D), ranks=(min(r[0], c["B"]),) + r[1:], cout=cout,
                 bf16=c["bf16"]) for _, D, cout, r in rows]


def dy_shape(layer):
    d = layer["dims"]
    if layer["kind"] == "linear":
        return d[:-1] + (layer["cout"],)
    out = [(n + 2 * layer["pad"] - layer["k"]) // layer["stride"] + 1 for n in d[2:]]
    return (d[0], layer["cout"], out[0], out[1])


def _inputs(layer, gen):
    """(activation, output gradient, previous factors) of one layer, on the GPU."""
    def normal(*shape):
        return torch.randn(*shape, generator=gen, device="cuda")

    dims, ranks = layer["dims"], layer["ranks"]
    tokens = layer["kind"] == "linear"
    # generating ranks and decay per index: 0.7 for the short conv ranks, scaled to the rank for wide token factors
    # (both factors of a matrix share one spectrum, so each takes half the decay)
    gr = [min(d, (2 if len(dims) > 2 else 3) * r if tokens else 24) for d, r in zip(dims, ranks)]
    rho = [0.7 ** ((8.0 if len(dims) > 2 else 3.0) / max(r, 8)) if tokens else 0.7 for r in ranks]
    act = normal(*gr)
    for m, (g, p) in enumerate(zip(gr, rho)):
        act *= (p ** torch.arange(g, device="cuda", dtype=torch.float32)).view([-1 if j == m else 1 for j in range(len(gr))])
    prev = []
    for m, (d, g, r) in enumerate(zip(dims, gr, ranks)):
        U = torch.linalg.qr(normal(d, g))[0]
        prev.append(torch.linalg.qr(U[:, :r] + 0.01 / math.sqrt(d) * normal(d, r))[0].reshape(-1))
        act = torch.movedim(torch.tensordot(U, act, dims=([1], [m])), 0, m)
    act = act / act.square().mean().sqrt() + 1e-3 * normal(*dims)
    shape = dy_shape(layer)
    dy = normal(*shape) / math.sqrt(math.prod(shape) / layer["cout"])
    dtype = torch.bfloat16 if layer["bf16"] else torch.float32
    return act.to(dtype).contiguous(), dy.to(dtype).contiguous(), torch.cat(prev)


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    s = dict(kind=case["kind"], seed=seed, runners=[], acts=[], dys=[])
    for layer in layers_of(case):
        act, dy, prev = _inputs(layer, gen)
        if case["kind"] == "host":
            run = LayerRunner(**layer)
            info = run.plan.info
            s["host_in"] = [x.cpu().pin_memory() for x in (act, dy, prev)]
            s["host_out"] = [torch.zeros(n, dtype=torch.float32).pin_memory()
                             for n in (info.u_elems, info.core_elems, info.dw_elems)]
            s["arena"] = torch.zeros(run.plan.step_host_arena_bytes(), dtype=torch.uint8, device="cuda")
        else:
            run = LayerRunner(**layer)
            run.U[run.cur].copy_(prev)
        s["runners"].append(run)
        s["acts"].append(act)
        s["dys"].append(dy)
    if case["kind"] == "step":
        s["step"] = StepRunner(s["runners"])
    return s


def run(state):
    rs = state["runners"]
    if state["kind"] == "host":
        # a device-resident caller would use the runner; this one keeps everything in pinned host memory
        a, d, u = state["host_in"]
        U, core, dW = state["host_out"]
        rs[0].plan.step_host(a.data_ptr(), d.data_ptr(), u.data_ptr(), U.data_ptr(), core.data_ptr(), dW.data_ptr(),
                             state["arena"].data_ptr(), state["arena"].numel(),
                             torch.cuda.current_stream().cuda_stream)
        return [U, core, dW]
    if state["kind"] == "cold":
        rs[0].init_factors_seeded(state["acts"][0], state["seed"])
        return [rs[0].U[rs[0].cur], rs[0].core]
    if state["kind"] == "step":
        state["step"].compress(state["acts"])
        state["step"].wgrad(state["dys"])
    else:
        rs[0].compress(state["acts"][0])
        rs[0].wgrad(state["dys"][0])
    return [x for r in rs for x in (r.U[r.cur], r.core, r.dW)]


def work(case):
    """Bytes: activation, output gradient and previous factors in; factors, core and weight gradient out.  Flops: two
    products per mode, the core products, and the weight gradient from the factors, two per multiply-add."""
    nbytes = flops = 0.0
    cold = case["kind"] == "cold"
    for layer in layers_of(case):
        eb = 2 if layer["bf16"] else 4
        dims, r, cout = layer["dims"], layer["ranks"], layer["cout"]
        n, dy = math.prod(dims), math.prod(dy_shape(layer))
        u, core = sum(d * x for d, x in zip(dims, r)), math.prod(r)
        macs = (1 if cold else 2) * n * sum(r)
        lead, rest = 1, n
        for d, x in zip(dims, r):
            macs += lead * rest * x
            lead, rest = lead * x, rest // d
        nbytes += n * eb + 4 * (u + core)
        if not cold:
            if layer["kind"] == "conv":
                k2, dw = layer["k"] ** 2, cout * (dims[1] // layer["groups"]) * layer["k"] ** 2
                macs += r[0] * dy + r[0] * r[1] * (r[2] * r[3] * dims[2] + r[3] * dims[2] * dims[3])
                macs += r[0] * r[1] * (dy // dims[0]) * k2 + r[1] * dw
            else:
                dw, z, lead = cout * dims[-1], dy, 1
                for d, x in zip(dims[:-1], r[:-1]):
                    macs += lead * z * x
                    lead, z = lead * x, z // d
                macs += lead * r[-1] * cout + r[-1] * dw
            nbytes += dy * eb + 4 * (u + dw)
        flops += 2.0 * macs
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    # sums are 32-bit or wider whatever the input type.  One step multiplies their rounding by the squared ratio of the
    # largest to the smallest kept singular value of a mode: tens for the conv ranks, some thousands for the widest
    # token factors; single entries of the weakest columns are further off than the whole.
    tokens = case["kind"] == "linear" or (case["kind"] == "step" and STEPS[case["layers"]][0] == "linear")
    return {"rel": 1e-4, "max": 2e-3} if tokens else {"rel": 3e-5, "max": 1e-3}
