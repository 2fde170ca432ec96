"""asi_compress_batched / asi_wgrad_batched: the layers of one training step in one call each way.
The batched calls must give the bits that one call per layer gives, and match the fp64 oracle."""
import threading

import numpy as np
import pytest
import torch

from asi_inputs.configs import LayerSpec, get_config, make_stream
from asi_inputs.generator import LayerStream
from oracle import asi_oracle as O
from tests.gpu_util import TOL_F32, make_runner, oracle_wgrad

pytestmark = pytest.mark.gpu


def _flat(U_list):
    return np.concatenate([np.ascontiguousarray(u, dtype=np.float32).ravel() for u in U_list])


def _check_batch(specs, streams, bf16=False, oracle_layers=()):
    from paper_2505_05086_b200.runner import StepRunner
    single = [make_runner(L, bf16=bf16) for L in specs]
    batched = [make_runner(L, bf16=bf16) for L in specs]
    step = StepRunner(batched)
    U0 = [st.u_prev0() for st in streams]
    for r, b, u in zip(single, batched, U0):
        r.set_factors(u)
        b.set_factors(u)
    for t in range(2):
        inputs = [st.next() for st in streams]
        acts = [r.to_device(A) for r, (A, _) in zip(single, inputs)]
        dys = [r.to_device(dY) for r, (_, dY) in zip(single, inputs)]
        for r, a, d in zip(single, acts, dys):
            r.compress(a)
            r.wgrad(d)
        step.compress(acts)
        step.wgrad(dys)
        torch.cuda.synchronize()
        for li, (r, b) in enumerate(zip(single, batched)):
            assert b.ok()
            assert torch.equal(r.U[r.cur], b.U[b.cur]), (t, li)
            assert torch.equal(r.core, b.core), (t, li)
            assert torch.equal(r.dW, b.dW), (t, li)
        if t == 0:
            for li in oracle_layers:
                L, (A, dY) = specs[li], inputs[li]
                S_ref, U_ref = O.asi_compress(A.astype(np.float64), [u.astype(np.float64) for u in U0[li]])
                dW_ref = oracle_wgrad(L, S_ref, U_ref, dY.astype(np.float64))
                U_gpu = batched[li].factors()
                assert max(O.rel_fro(O.projector(a), O.projector(b)) for a, b in zip(U_gpu, U_ref)) <= TOL_F32["proj"]
                assert O.rel_fro(batched[li].dW_np(L.dw_shape), dW_ref) <= TOL_F32["dw"]


def test_resnet18_last4_step_in_two_calls():
    cfg = get_config(1)          # three 7x7 layers and one 14x14 layer: two kernel variants
    _check_batch(list(cfg.layers), [make_stream(cfg, li) for li in range(4)], oracle_layers=(0, 3))


def test_mobilenetv2_last5_step_in_two_calls():
    cfg = get_config(2)          # five 7x7 layers (one depthwise), one variant: 3 + 1 launches for the step
    _check_batch(list(cfg.layers), [make_stream(cfg, li) for li in range(5)], oracle_layers=(2,))


def test_mixed_batch_fused_generic_and_linear_layers():
    specs = [LayerSpec("a", "conv", (8, 12, 7, 7), 10, 3, 1, 1, 1, ranks=(3, 4, 3, 2)),
             LayerSpec("b", "conv", (5, 12, 9, 11), 7, 3, 1, 1, 1, ranks=(3, 5, 4, 6)),       # generic kernels
             LayerSpec("c", "linear", (6, 37, 50), 21, ranks=(3, 5, 7)),
             LayerSpec("d", "conv", (16, 20, 7, 7), 12, 1, 1, 0, 1, ranks=(5, 8, 4, 4)),       # the rank 5..8 variant
             LayerSpec("e", "conv", (8, 16, 7, 7), 16, 3, 1, 1, 16, ranks=(2, 3, 3, 3))]       # depthwise, same variant as a
    streams = [LayerStream(dims=L.dims, ranks=L.ranks, dy_shape=L.dy_shape, seed=90 + i,
                           rho=tuple(min(0.7, 0.25 ** (1.0 / max(r - 1, 1))) for r in L.ranks),
                           gen_ranks=tuple(min(d, max(r + 2, 4)) for d, r in zip(L.dims, L.ranks)))
               for i, L in enumerate(specs)]
    _check_batch(specs, streams, oracle_layers=(0, 1, 2, 3, 4))


def _random_layers(specs, seed):
    """Runners with random orthonormal factors, and random inputs (no oracle: single calls are the reference)."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    runs, acts, dys = [], [], []
    for L in specs:
        r = make_runner(L)
        r.set_factors([torch.linalg.qr(torch.randn(d, k, generator=gen, device="cuda"))[0].cpu().numpy()
                       for d, k in zip(L.dims, L.ranks)])
        runs.append(r)
        acts.append(torch.randn(*L.dims, generator=gen, device="cuda"))
        dys.append(torch.randn(*L.dy_shape, generator=gen, device="cuda"))
    return runs, acts, dys


SHARING = [LayerSpec("a", "conv", (8, 24, 28, 28), 40, 3, 1, 1, 1, ranks=(3, 4, 3, 4)),      # four launches, split Z4
           LayerSpec("b", "conv", (8, 24, 30, 26), 24, 3, 1, 1, 1, ranks=(4, 5, 6, 4)),
           LayerSpec("c", "linear", (6, 37, 50), 21, ranks=(3, 5, 7)),
           LayerSpec("d", "conv", (8, 12, 7, 7), 10, 3, 1, 1, 1, ranks=(3, 4, 3, 2)),        # fused
           LayerSpec("e", "conv", (8, 16, 7, 7), 16, 3, 1, 1, 1, ranks=(2, 3, 3, 3))]


@pytest.mark.parametrize("which", ["workspace", "overlap", "gradient"])
def test_wgrad_layers_that_share_memory_run_one_after_another(which):
    """One workspace for all layers, workspaces that overlap in part, and layers of one shape with one dW: what separate
    calls give, twenty times over."""
    specs = SHARING if which != "gradient" else [SHARING[0]] * 3
    runs, acts, dys = _random_layers(specs, 7)
    want = []
    for r, a, d in zip(runs, acts, dys):
        r.compress(a)
        r.wgrad(d)
        want.append(r.dW.clone())
    from paper_2505_05086_b200.runner import StepRunner
    step = StepRunner(runs)
    most = max(r.ws_w.numel() for r in runs)
    arena = torch.zeros(most + 4096 * len(runs), dtype=torch.uint8, device="cuda")
    if which == "gradient":
        for r in runs[1:]:
            r.dW = runs[0].dW
    else:
        for i, r in enumerate(runs):
            at = 4096 * i if which == "overlap" else 0
            r.ws_w = arena[at:at + most]
    for _ in range(20):
        for r in runs:
            r.dW.fill_(float("nan"))
        step.wgrad(dys)
        torch.cuda.synchronize()
        if which == "gradient":
            assert torch.equal(runs[0].dW, want[-1])
        else:
            assert all(torch.equal(r.dW, w) for r, w in zip(runs, want))


def test_compress_layers_whose_workspaces_overlap_run_one_after_another():
    runs, acts, _ = _random_layers(SHARING, 8)
    want = []
    for r, a in zip(runs, acts):
        r.compress(a)
        want.append((r.U[r.cur].clone(), r.core.clone()))
        r.cur = 1 - r.cur
    from paper_2505_05086_b200.runner import StepRunner
    most = max(r.ws_c.numel() for r in runs)
    arena = torch.zeros(most + 4096 * len(runs), dtype=torch.uint8, device="cuda")
    for i, r in enumerate(runs):
        r.ws_c = arena[4096 * i:4096 * i + most]
    step = StepRunner(runs)
    for _ in range(20):
        step.compress(acts)
        torch.cuda.synchronize()
        for r, (u, c) in zip(runs, want):
            assert torch.equal(r.U[r.cur], u) and torch.equal(r.core, c)
            r.cur = 1 - r.cur


@pytest.mark.parametrize("bf16", [False, True])
def test_layers_of_a_group_with_shifted_activations(bf16):
    """Layers of one variant, two of which start at odd elements: they leave the shared launch, and every layer gives what
    its separate call gives."""
    from paper_2505_05086_b200.runner import StepRunner
    specs = [LayerSpec("a", "conv", (8, 12 + 4 * i, 7, 7), 12, 3, 1, 1, 1, ranks=(3, 4, 3, 2)) for i in range(4)]
    gen = torch.Generator(device="cuda").manual_seed(5)
    dtype = torch.bfloat16 if bf16 else torch.float32

    def shifted(shape, k):
        n = int(np.prod(shape))
        return torch.randn(n + 8, generator=gen, device="cuda").to(dtype)[k:k + n].view(shape)

    runs = [make_runner(L, bf16=bf16) for L in specs]
    acts = [shifted(L.dims, k) for L, k in zip(specs, (0, 1, 0, 3))]
    dys = [shifted(L.dy_shape, k) for L, k in zip(specs, (2, 0, 1, 0))]
    want = []
    for r, L, a, d in zip(runs, specs, acts, dys):
        r.set_factors([np.linalg.qr(np.random.default_rng(3).standard_normal((n, k)))[0] for n, k in zip(L.dims, L.ranks)])
        r.compress(a)
        r.wgrad(d)
        want.append((r.U[r.cur].clone(), r.core.clone(), r.dW.clone()))
        r.cur = 1 - r.cur
    step = StepRunner(runs)
    step.compress(acts)
    step.wgrad(dys)
    torch.cuda.synchronize()
    for r, w in zip(runs, want):
        assert all(torch.equal(x, y) for x, y in zip((r.U[r.cur], r.core, r.dW), w))


# Layers of few CTAs hold their tile in shared memory, steps of many CTAs stream it: the same bits.  Channels beyond the last
# whole tile, few samples, a batch that is no multiple of the shares, ranks of both buckets, rows of odd length (not staged)
FORMS = [
    ((10, 130, 6, 6), (4, 4, 4, 4), 20, 3),
    ((3, 84, 14, 14), (3, 3, 4, 4), 16, 3),
    ((70, 100, 7, 8), (4, 5, 4, 6), 12, 1),
    ((13, 133, 7, 7), (4, 4, 4, 3), 12, 3),
    ((130, 96, 7, 7), (3, 4, 3, 4), 24, 3),
]


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("case", FORMS)
def test_staged_and_streamed_tiles_give_the_same_bits(case, bf16):
    from paper_2505_05086_b200.runner import StepRunner
    dims, ranks, cout, k = case
    L = LayerSpec("t", "conv", dims, cout, k, 1, k // 2, 1, ranks=ranks)
    gen = torch.Generator(device="cuda").manual_seed(11)
    dtype = torch.bfloat16 if bf16 else torch.float32
    rng = np.random.default_rng(5)
    runs = [make_runner(L, bf16=bf16) for _ in range(16)]
    acts = [torch.randn(*dims, generator=gen, device="cuda").to(dtype) for _ in runs]
    dys = [torch.randn(*L.dy_shape, generator=gen, device="cuda").to(dtype) for _ in runs]
    want = []
    for r, a, d in zip(runs, acts, dys):
        r.set_factors([np.linalg.qr(rng.standard_normal((n, q)))[0] for n, q in zip(dims, ranks)])
        r.compress(a)
        r.wgrad(d)
        want.append((r.U[r.cur].clone(), r.core.clone(), r.dW.clone()))
        r.cur = 1 - r.cur
    step = StepRunner(runs)
    step.compress(acts)
    step.wgrad(dys)
    torch.cuda.synchronize()
    for r, w in zip(runs, want):
        assert r.ok()
        assert all(torch.equal(x, y) for x, y in zip((r.U[r.cur], r.core, r.dW), w))


# twelve chains (no two layers share launches): more than a call has side streams
MANY = [LayerSpec("c%d" % i, "conv", (6 + i, 9 + i, 18 + i, 21), 8 + i, 3, 1, 1, 1, ranks=(3, 4, 3, 4)) for i in range(6)] + \
       [LayerSpec("l%d" % i, "linear", (5 + i, 33, 40 + 8 * i), 20 + i, ranks=(3, 5, 7)) for i in range(6)]


def _singles(runs, acts, dys):
    out = []
    for r, a, d in zip(runs, acts, dys):
        r.compress(a)
        r.wgrad(d)
        out.append((r.U[r.cur].clone(), r.core.clone(), r.dW.clone()))
        r.cur = 1 - r.cur
    torch.cuda.synchronize()
    return out


def _same(runs, want):
    return all(torch.equal(x, y) for r, w in zip(runs, want) for x, y in zip((r.U[r.cur], r.core, r.dW), w))


def test_more_chains_than_side_streams():
    from paper_2505_05086_b200.runner import StepRunner
    runs, acts, dys = _random_layers(MANY, 21)
    want = _singles(runs, acts, dys)
    step = StepRunner(runs)
    for _ in range(5):
        step.compress(acts)
        step.wgrad(dys)
        torch.cuda.synchronize()
        assert _same(runs, want)
        for r in runs:
            r.cur = 1 - r.cur


@pytest.mark.parametrize("specs", [SHARING, MANY])
def test_batched_calls_in_a_captured_graph(specs):
    """Captured on one stream: the layers follow one another there, the side streams stay out of the capture and serve
    calls outside it while the graph exists."""
    from paper_2505_05086_b200.runner import StepRunner
    runs, acts, dys = _random_layers(specs, 22)
    want = _singles(runs, acts, dys)
    step = StepRunner(runs)
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        step.compress(acts)                          # warm
        step.wgrad(dys)
        for r in runs:
            r.cur = 1 - r.cur
        stream.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            step.compress(acts)
            step.wgrad(dys)
    for _ in range(3):
        for r in runs:
            r.dW.zero_()
            r.core.zero_()
            r.U[r.cur].zero_()
        torch.cuda.synchronize()
        graph.replay()
        torch.cuda.synchronize()
        assert _same(runs, want)
    for r in runs:
        r.cur = 1 - r.cur
    step.compress(acts)
    step.wgrad(dys)
    torch.cuda.synchronize()
    assert _same(runs, want)
    del graph


def test_batched_calls_from_several_host_threads():
    """Ten threads with layers and a stream of their own: more callers at a time than there are sets of side streams."""
    from paper_2505_05086_b200.runner import StepRunner
    specs = [MANY[0], MANY[7], SHARING[3], SHARING[4], SHARING[0]]
    jobs = []
    for i in range(10):
        runs, acts, dys = _random_layers(specs, 30 + i)
        jobs.append((runs, acts, dys, _singles(runs, acts, dys), torch.cuda.Stream()))
    torch.cuda.synchronize()
    errors = []
    start = threading.Barrier(len(jobs))

    def work(runs, acts, dys, want, stream):
        try:
            step = StepRunner(runs)
            start.wait(timeout=60)
            for _ in range(25):
                step.compress(acts, stream)
                step.wgrad(dys, stream)
                stream.synchronize()
                if not _same_on(stream, runs, want):
                    raise AssertionError("results differ")
                for r in runs:
                    r.cur = 1 - r.cur
        except BaseException as e:                   # handed to the test's own thread
            errors.append(e)

    def _same_on(stream, runs, want):
        with torch.cuda.stream(stream):
            return _same(runs, want)

    threads = [threading.Thread(target=work, args=j) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join(timeout=120)
    assert not errors, errors
    assert not any(t.is_alive() for t in threads)


@pytest.mark.parametrize("spec,bf16", [
    (LayerSpec("fused", "conv", (16, 24, 14, 14), 20, 3, 1, 1, 1, ranks=(4, 4, 4, 4)), False),
    (LayerSpec("clustered", "conv", (136, 20, 7, 7), 12, 3, 1, 1, 1, ranks=(4, 4, 4, 4)), False),
    (LayerSpec("large", "conv", (32, 64, 28, 28), 40, 3, 1, 1, 1, ranks=(4, 4, 4, 4)), False),
    (LayerSpec("planes", "conv", (16, 40, 56, 56), 40, 3, 1, 1, 1, ranks=(4, 4, 4, 4)), True),
    (LayerSpec("tokens", "linear", (16, 40, 128), 64, ranks=(8, 12, 16)), True),
    (LayerSpec("matrix", "linear", (64, 300), 64, ranks=(12, 12)), False),
], ids=lambda p: getattr(p, "name", str(p)))
def test_calls_captured_behind_a_join_of_two_streams(spec, bf16):
    """The first kernel of a call depends on two nodes of the graph, one of them on another stream; it must wait for both: the
    activation and the gradient are written by these, anew in each replay."""
    run = make_runner(spec, bf16=bf16)
    gen = torch.Generator(device="cuda").manual_seed(11)

    def normal(shape):
        return torch.randn(*shape, generator=gen, device="cuda").to(run.in_dtype)

    a_src, d_src = normal(spec.dims), normal(spec.dy_shape)
    act, dy, prev = torch.zeros_like(a_src), torch.zeros_like(d_src), torch.zeros_like(run.U[0])
    u_src = torch.cat([torch.linalg.qr(torch.randn(d, r, generator=gen, device="cuda"))[0].reshape(-1)
                       for d, r in zip(spec.dims, spec.ranks)])
    main, side = torch.cuda.Stream(), torch.cuda.Stream()

    def enqueue():
        side.wait_stream(main)
        with torch.cuda.stream(side):
            torch.mul(u_src, 1.0, out=run.U[0])
        torch.mul(a_src, 0.5, out=act)
        main.wait_stream(side)
        run.cur = 0
        run.compress(act, stream=main)
        side.wait_stream(main)
        with torch.cuda.stream(side):
            torch.mul(d_src, 0.5, out=dy)
        torch.mul(prev, 0.5, out=prev)
        main.wait_stream(side)
        run.wgrad(dy, stream=main)

    with torch.cuda.stream(main):
        enqueue()                                    # loads the kernels
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=main):
        enqueue()
    for _ in range(3):
        a_src.copy_(normal(spec.dims))
        d_src.copy_(normal(spec.dy_shape))
        out = []
        for replay in (True, False):
            for x in (act, dy, run.U[0], run.U[1], run.core, run.dW):
                x.zero_()
            torch.cuda.synchronize()
            if replay:
                graph.replay()
            else:
                with torch.cuda.stream(main):
                    enqueue()
            torch.cuda.synchronize()
            assert run.ok()
            out.append([x.clone() for x in (run.U[1], run.core, run.dW)])
        assert all(float(x.abs().sum()) > 0 for x in out[0])
        assert all(torch.equal(x, y) for x, y in zip(*out))
