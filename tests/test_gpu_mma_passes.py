"""Mode passes with the factor on the tensor cores, at the sizes where their tiling can go wrong, against the fp64 oracle
and the shape-generic kernels."""
import numpy as np
import pytest
import torch

from asi_inputs.configs import LayerSpec
from asi_inputs.generator import LayerStream
from oracle import asi_oracle as O
from tests.gpu_util import TOL_F32, check, compare_step, make_runner

pytestmark = pytest.mark.gpu

CASES = [  # (dims, ranks, bf16)
    ((17, 33, 17, 20), (3, 4, 4, 4), False),       # two row tiles and one row more; columns in whole quads
    ((65, 16, 18, 19), (4, 4, 3, 2), False),       # two warps a tile, the second nearly empty; odd rows
    ((12, 130, 17, 17), (5, 8, 6, 7), False),      # three warps a tile, ranks above four, odd planes
    ((6, 257, 16, 20), (2, 3, 4, 4), False),       # five warps a tile
    ((3, 384, 17, 16), (3, 6, 5, 3), False),       # the longest mode, six warps
    ((2, 48, 32, 32), (2, 4, 4, 4), False),        # the largest planes, a batch of two
    ((16, 10, 12, 24), (4, 4, 4, 4), False),       # the smallest planes of their kernel, one row tile
    ((9, 40, 31, 13), (4, 5, 8, 8), False),        # no square, no multiple of anything
    ((128, 8, 28, 28), (3, 3, 3, 3), False),       # a full team; planes of 28
    ((40, 48, 24, 24), (4, 4, 4, 4), True),        # bf16 rows and planes on 16 bytes
    ((33, 128, 20, 20), (6, 5, 7, 5), True),       # bf16, ranks above four: 32 rows a warp
    ((16, 24, 18, 26), (3, 4, 4, 4), True),        # bf16 rows off 16 bytes: the kernels of any address
]


@pytest.mark.parametrize("dims,ranks,bf16", CASES)
def test_mode_passes_against_the_oracle_and_the_generic_kernels(dims, ranks, bf16):
    # decay that keeps sigma_r / sigma_1 >= 0.25, as the other small cases have it: fp32 sums then stay far below 1e-4
    rho = tuple(min(0.7, 0.25 ** (1.0 / max(r - 1, 1))) for r in ranks)
    L = LayerSpec("t", "conv", dims, 6, 3, 1, 1, 1, ranks=ranks)
    st = LayerStream(dims=dims, ranks=ranks, dy_shape=L.dy_shape, seed=sum(dims), rho=rho, bf16=bf16,
                     gen_ranks=tuple(min(d, max(r + 2, 4)) for d, r in zip(dims, ranks)))
    run, gen = make_runner(L, bf16=bf16), make_runner(L, bf16=bf16, generic_only=True)
    U_prev = st.u_prev0()
    for t in range(2):
        A, dY = st.next()
        err_g, _ = compare_step(gen, L, A, dY, U_prev)
        err, U_prev = compare_step(run, L, A, dY, U_prev)
        check(err_g, TOL_F32, f"generic {dims}")
        check(err, TOL_F32, str(dims))


@pytest.mark.parametrize("dims,ranks", [((50, 116, 27, 27), (5, 6, 5, 5)), ((40, 40, 18, 21), (5, 5, 6, 8))])
def test_any_element_address(dims, ranks):
    """Layers that take an fp32 activation at any element: off 16 bytes its rows and planes come by four-byte copies.  The sums
    are the same up to the order of fp32 additions (1e-6 on well-conditioned random data, times ten)."""
    L = LayerSpec("t", "conv", dims, 6, 3, 1, 1, 1, ranks=ranks)
    run = make_runner(L)
    rng = np.random.default_rng(3)
    A = torch.from_numpy(rng.standard_normal(dims).astype(np.float32)).cuda()
    run.U[0].copy_(torch.randn(run.plan.info.u_elems, generator=torch.Generator().manual_seed(1)))
    big = torch.zeros(A.numel() + 8, device="cuda")
    out = []
    for shift in (0, 1, 3):
        big[shift:shift + A.numel()].copy_(A.reshape(-1))
        run.cur = 0
        run.compress(big[shift:shift + A.numel()])
        torch.cuda.synchronize()
        assert run.ok()
        out.append([run.U[1].clone(), run.core.clone()])
    for o in out[1:]:
        for x, y in zip(o, out[0]):
            assert float((x - y).norm() / y.norm()) <= 1e-5


TOKENS = [  # (dims, ranks, cout, bf16): batches on both sides of the rule's line and of a tile
    ((8, 40, 128), (4, 12, 16), 24, True),
    ((9, 40, 128), (8, 12, 16), 24, True),
    ((17, 33, 96), (4, 8, 12), 20, False),
    ((33, 24, 130), (7, 8, 12), 20, False),        # rows off 16 bytes
    ((130, 24, 64), (5, 8, 8), 20, False),         # three warps a tile
]


@pytest.mark.parametrize("dims,ranks,cout,bf16", TOKENS)
def test_batch_mode_of_token_layers(dims, ranks, cout, bf16):
    rho = tuple(min(0.95, 0.25 ** (1.0 / max(r - 1, 1))) for r in ranks)
    L = LayerSpec("t", "linear", dims, cout, ranks=ranks)
    st = LayerStream(dims=dims, ranks=ranks, dy_shape=L.dy_shape, seed=sum(dims), rho=rho, bf16=bf16,
                     gen_ranks=tuple(min(d, 2 * r) for d, r in zip(dims, ranks)))
    run = make_runner(L, bf16=bf16)
    U_prev = st.u_prev0()
    for t in range(2):
        A, dY = st.next()
        err, U_prev = compare_step(run, L, A, dY, U_prev)
        check(err, TOL_F32, str(dims))


@pytest.mark.parametrize("dims,ranks,bf16", [c for c in CASES if c[0][0] >= 6])
def test_cold_start_passes(dims, ranks, bf16):
    """P_m = A_m Omega_m of the same layers (1e-4 as everywhere; the spectra keep the iterate's condition number below a hundred).
    They are below a million values, so SIMT products do it; the passes with Omega in place of V are tested on larger ones."""
    rho = tuple(min(0.7, 0.25 ** (1.0 / max(r - 1, 1))) for r in ranks)
    L = LayerSpec("t", "conv", dims, 6, 3, 1, 1, 1, ranks=ranks)
    st = LayerStream(dims=dims, ranks=ranks, dy_shape=L.dy_shape, seed=sum(dims), rho=rho, bf16=bf16,
                     gen_ranks=tuple(min(d, max(r + 2, 4)) for d, r in zip(dims, ranks)))
    A, _ = st.next()
    rng = np.random.default_rng(5)
    n = int(np.prod(dims))
    Omega = [rng.standard_normal((n // d, r)).astype(np.float32) for d, r in zip(dims, ranks)]
    run = make_runner(L, bf16=bf16)
    run.init_factors(run.to_device(A), torch.from_numpy(np.concatenate([o.ravel() for o in Omega])).cuda())
    assert run.ok()
    S_ref, U_ref = O.asi_cold_start(A.astype(np.float64), [o.astype(np.float64) for o in Omega])
    U = run.factors()
    assert max(O.rel_fro(O.projector(a), O.projector(b)) for a, b in zip(U, U_ref)) <= 1e-4
    assert O.rel_fro(O.sign_align(run.core_np(), U, U_ref)[0], S_ref) <= 1e-4


WGRADS = [  # (dims, cout, k, stride, groups, ranks, split launches): both sides of the rule's three lines
    ((16, 24, 24, 24), 24, 3, 1, 1, (3, 4, 4, 4), True),       # 9216 values a CTA
    ((14, 24, 24, 24), 24, 3, 1, 1, (3, 4, 4, 4), False),      # 8064: one CTA a channel
    ((13, 30, 25, 27), 148, 3, 1, 1, (4, 4, 4, 4), True),      # as many channels as SMs; odd planes of dY
    ((13, 30, 25, 27), 149, 3, 1, 1, (4, 4, 4, 4), False),
    ((40, 24, 29, 29), 36, 3, 2, 12, (4, 4, 4, 4), True),      # grouped, strided
    ((16, 20, 24, 24), 20, 5, 1, 20, (4, 8, 8, 8), True),      # depthwise
    ((16, 24, 24, 24), 24, 1, 1, 1, (4, 4, 4, 4), False),      # 1 x 1
]


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("dims,cout,k,stride,groups,ranks,split", WGRADS)
def test_weight_gradient_routes_of_large_maps(dims, cout, k, stride, groups, ranks, split, bf16):
    """dY at a sixteen-byte address and one element past it, on either side of the line between the launches."""
    rho = tuple(min(0.7, 0.25 ** (1.0 / max(r - 1, 1))) for r in ranks)
    L = LayerSpec("t", "conv", dims, cout, k, stride, k // 2, groups, ranks=ranks)
    st = LayerStream(dims=dims, ranks=ranks, dy_shape=L.dy_shape, seed=sum(dims), rho=rho, bf16=bf16,
                     gen_ranks=tuple(min(d, max(r + 2, 4)) for d, r in zip(dims, ranks)))
    run = make_runner(L, bf16=bf16)
    assert (run.plan.launch_count(1) > 1) == split
    A, dY = st.next()
    U_prev = st.u_prev0()
    to_device = run.to_device
    for shift in (0, 1):
        def place(x):
            t = to_device(x)
            if x is A:
                return t
            buf = torch.full((t.numel() + 8,), float("nan"), dtype=t.dtype, device=t.device)
            view = buf[shift:shift + t.numel()].view(t.shape)
            view.copy_(t)
            return view

        run.to_device = place
        err, _ = compare_step(run, L, A, dY, U_prev)
        check(err, TOL_F32, f"{dims} {cout} bf16={bf16} shift={shift}")


NAN_BITS = 0x7fffffff                              # the NaN that arithmetic on the GPU makes
NANS = [c for c in CASES if c[0] in ((17, 33, 17, 20), (12, 130, 17, 17), (40, 48, 24, 24), (33, 128, 20, 20))]


def _put_nan(flat, at):
    flat.view(torch.int32)[at] = NAN_BITS


@pytest.mark.parametrize("dims,ranks,bf16", NANS)
def test_a_nan_in_a_factor_reaches_the_results(dims, ranks, bf16):
    """One NaN in column 1 of U_m (or of Omega_m): that column of P_m and so every column of the new factor from there on, and with
    the core all of the gradient."""
    from paper_2505_05086_b200.binding import ASI_ERR_RANK_DEFICIENT
    L = LayerSpec("t", "conv", dims, 6, 3, 1, 1, 1, ranks=ranks)
    run = make_runner(L, bf16=bf16)
    rng = np.random.default_rng(4)
    act, dY = (run.to_device(rng.standard_normal(s)) for s in (dims, L.dy_shape))
    U0 = np.concatenate([np.linalg.qr(rng.standard_normal((d, r)))[0].ravel() for d, r in zip(dims, ranks)])
    n = int(np.prod(dims))
    omega = torch.from_numpy(rng.standard_normal(sum(n // d * r for d, r in zip(dims, ranks))).astype(np.float32)).cuda()
    at_u = at_o = 0
    for m, (d, r) in enumerate(zip(dims, ranks)):
        for cold in (False, True):
            if cold:
                om = omega.clone()
                _put_nan(om, at_o + (n // d // 2) * r + 1)
                run.init_factors(act, om)
            else:
                run.U[run.cur].copy_(torch.from_numpy(U0.astype(np.float32)))
                _put_nan(run.U[run.cur], at_u + (d // 2) * r + 1)
                run.compress(act)
            run.wgrad(dY)
            assert run.device_status() == ASI_ERR_RANK_DEFICIENT, (m, cold)
            U = run.factors()
            assert np.isnan(U[m][:, 1:]).all(), (m, cold)
            assert all(np.isfinite(u).all() for q, u in enumerate(U) if q != m), (m, cold)
            assert np.isnan(np.moveaxis(run.core_np(), m, 0)[1:]).all(), (m, cold)
            assert np.isnan(run.dW.cpu().numpy()).all(), (m, cold)
        at_u += d * r
        at_o += n // d * r


@pytest.mark.parametrize("dims,ranks,bf16", NANS)
def test_a_nan_in_the_activation_stays_in_the_factors_of_the_next_step(dims, ranks, bf16):
    L = LayerSpec("t", "conv", dims, 6, 3, 1, 1, 1, ranks=ranks)
    run = make_runner(L, bf16=bf16)
    rng = np.random.default_rng(4)
    act, dY = (run.to_device(rng.standard_normal(s)) for s in (dims, L.dy_shape))
    run.set_factors([np.linalg.qr(rng.standard_normal((d, r)))[0] for d, r in zip(dims, ranks)])
    bad = act.clone()
    bad.view(-1)[act.numel() // 2] = float("nan")
    for x in (bad, act):
        run.compress(x)
        run.wgrad(dY)
        assert not run.ok()
        assert all(np.isnan(u).all() for u in run.factors())
        assert np.isnan(run.dW.cpu().numpy()).all()


@pytest.mark.parametrize("dims,ranks,cout,bf16", TOKENS[1:])
def test_a_nan_in_the_batch_factor_of_a_token_layer(dims, ranks, cout, bf16):
    L = LayerSpec("t", "linear", dims, cout, ranks=ranks)
    run = make_runner(L, bf16=bf16)
    rng = np.random.default_rng(4)
    run.set_factors([np.linalg.qr(rng.standard_normal((d, r)))[0] for d, r in zip(dims, ranks)])
    _put_nan(run.U[run.cur], dims[0] // 2 * ranks[0] + 1)
    run.compress(run.to_device(rng.standard_normal(dims)))
    run.wgrad(run.to_device(rng.standard_normal(L.dy_shape)))
    assert not run.ok()
    assert np.isnan(run.factors()[0][:, 1:]).all()
    assert np.isnan(run.dW.cpu().numpy()).all()


@pytest.mark.parametrize("dims,ranks,bf16", NANS)
def test_a_factor_of_the_largest_values(dims, ranks, bf16):
    """U_m scaled to the top of fp32 beside an activation scaled down: the same factor as without (1e-6 of rounding on
    well-conditioned random data, times ten)."""
    L = LayerSpec("t", "conv", dims, 6, 3, 1, 1, 1, ranks=ranks)
    run = make_runner(L, bf16=bf16)
    rng = np.random.default_rng(4)
    act = run.to_device(rng.standard_normal(dims))
    U0 = [np.linalg.qr(rng.standard_normal((d, r)))[0].astype(np.float32) for d, r in zip(dims, ranks)]
    out = []
    for scale in (1.0, 2.0 ** -60):
        U = [u.copy() for u in U0]
        for u in U:
            u[:] = np.sign(u) * (1.0 if scale == 1.0 else np.finfo(np.float32).max)
        run.set_factors(U)
        run.compress(act * scale)
        assert run.ok()
        out.append(run.factors())
    for a, b in zip(*out):
        assert np.linalg.norm(a - b) / np.linalg.norm(b) <= 1e-5


@pytest.mark.parametrize("cold", [False, True])
@pytest.mark.parametrize("kind,dims,ranks,bf16", [
    ("conv", (16, 130, 28, 28), (4, 4, 4, 4), False),          # planes, and teams of one and of three warps
    ("conv", (16, 130, 40, 40), (5, 6, 5, 5), False),          # strided fibers alone
    ("conv", (40, 48, 24, 24), (4, 4, 4, 4), True),
    ("conv", (16, 48, 56, 56), (4, 4, 4, 4), False),           # the planes of their own kernel
    ("linear", (33, 64, 1024), (7, 8, 12), True),
    ("linear", (8, 64, 256), (4, 16, 16), True),               # tcgen05 products: one tile a CTA, and tiles shared by a cluster
    ("linear", (24, 128, 1664), (4, 16, 16), True),            # several tiles a CTA
])
def test_expired_waits_are_reported_and_the_workspace_recovers(kind, dims, ranks, bf16, cold):
    """The producer arms its barriers and copies nothing; every wait runs out (1 ms), and the next call on the same workspace is
    healthy again."""
    from paper_2505_05086_b200.binding import ASI_ERR_TIMEOUT, ASI_FLAG_TEST_EXPIRE_WAIT, Plan
    L = LayerSpec("t", kind, dims, 10, 3, 1, 1, 1, ranks=ranks) if kind == "conv" else LayerSpec("t", kind, dims, 10, ranks=ranks)
    rho = tuple(min(0.95, 0.25 ** (1.0 / max(r - 1, 1))) for r in ranks)
    st = LayerStream(dims=dims, ranks=ranks, dy_shape=L.dy_shape, seed=7, rho=rho, bf16=bf16,
                     gen_ranks=tuple(min(d, 2 * r) for d, r in zip(dims, ranks)))
    A, dY = st.next()
    run = make_runner(L, bf16=bf16)
    stalled = Plan(kind, dims, ranks, 10, L.k, L.stride, L.pad, L.groups, bf16, flags=ASI_FLAG_TEST_EXPIRE_WAIT)
    assert stalled.info.compress_ws_bytes == run.plan.info.compress_ws_bytes
    U_prev = st.u_prev0()
    run.set_factors(U_prev)
    act = run.to_device(A)
    s = int(torch.cuda.current_stream().cuda_stream)
    out = [run.U[1 - run.cur].data_ptr(), run.core.data_ptr(), run.ws_c.data_ptr(), run.ws_c.numel(), s]
    if cold:
        n = int(np.prod(dims))
        omega = torch.randn(sum(n // d * r for d, r in zip(dims, ranks)), device="cuda")
        stalled.init_factors(act.data_ptr(), omega.data_ptr(), *out)
    else:
        stalled.compress(act.data_ptr(), run.U[run.cur].data_ptr(), *out)
    assert stalled.poll_status(run.ws_c.data_ptr(), s) == ASI_ERR_TIMEOUT
    err, _ = compare_step(run, L, A, dY, U_prev)
    check(err, TOL_F32, f"{dims} after an expired wait")
    assert run.device_status() == 0


@pytest.mark.parametrize("dims,ranks,bf16", [((28, 92, 28, 28), (6, 8, 5, 8), True), ((11, 300, 56, 28), (1, 7, 5, 4), False),
                                             ((9, 274, 24, 24), (2, 8, 12, 8), False)])
def test_built_in_workspace(dims, ranks, bf16):
    """Layers near its 4 MiB, whose scratch regions take one another's place: the same bits as with a workspace of the caller's,
    whatever it held before."""
    L = LayerSpec("t", "conv", dims, 6, 3, 1, 1, 1, ranks=ranks)
    run = make_runner(L, bf16=bf16)
    rng = np.random.default_rng(4)
    run.set_factors([np.linalg.qr(rng.standard_normal((d, r)))[0] for d, r in zip(dims, ranks)])
    act = run.to_device(rng.standard_normal(dims))
    run.ws_c.fill_(0xff)
    run.compress(act)
    assert run.ok()
    U, core = torch.empty_like(run.U[0]), torch.empty_like(run.core)
    for _ in range(2):
        run.plan.compress_static_ws(act.data_ptr(), run.U[0].data_ptr(), U.data_ptr(), core.data_ptr(),
                                    int(torch.cuda.current_stream().cuda_stream))
        assert torch.equal(U, run.U[1]) and torch.equal(core, run.core)


COLD = [  # (dims, ranks, bf16, launches of the passes): a million values with a pass for every mode, two million without
    ((65, 60, 18, 19), (4, 4, 3, 2), False, 3),    # two warps a tile along the batch; odd rows along the channels
    ((40, 130, 17, 17), (5, 8, 6, 7), False, 3),   # three warps, ranks above four, odd planes
    ((17, 200, 20, 20), (3, 4, 4, 4), False, 3),   # two row tiles and one row more
    ((12, 384, 17, 16), (3, 6, 5, 3), False, 3),   # the longest mode
    ((40, 48, 24, 24), (4, 4, 4, 4), True, 3),
    ((33, 128, 20, 20), (6, 5, 7, 5), True, 3),
    ((13, 25, 56, 60), (4, 4, 4, 4), False, 0),    # planes without a pass: below two million the SIMT products do it all
    ((30, 25, 56, 60), (4, 4, 4, 4), False, 2),
    ((11, 70, 36, 36), (4, 6, 4, 4), True, 0),
    ((9, 100, 24, 24), (4, 5, 4, 4), False, 0),    # a pass for every mode, half a million
    ((8, 260, 24, 24), (4, 5, 4, 4), False, 3),    # a batch of eight: half a row tile, and only here
    ((3, 120, 56, 60), (3, 5, 4, 4), False, 2),    # planes without a pass, but a batch below eight
]


@pytest.mark.parametrize("dims,ranks,bf16,passes", COLD)
def test_cold_start_on_both_sides_of_the_passes(dims, ranks, bf16, passes):
    import ctypes
    from paper_2505_05086_b200.binding import lib
    rho = tuple(min(0.7, 0.25 ** (1.0 / max(r - 1, 1))) for r in ranks)
    L = LayerSpec("t", "conv", dims, 6, 3, 1, 1, 1, ranks=ranks)
    st = LayerStream(dims=dims, ranks=ranks, dy_shape=L.dy_shape, seed=sum(dims), rho=rho, bf16=bf16,
                     gen_ranks=tuple(min(d, max(r + 2, 4)) for d, r in zip(dims, ranks)))
    A, _ = st.next()
    rng = np.random.default_rng(5)
    n = int(np.prod(dims))
    Omega = [rng.standard_normal((n // d, r)).astype(np.float32) for d, r in zip(dims, ranks)]
    run = make_runner(L, bf16=bf16)
    act, omega = run.to_device(A), torch.from_numpy(np.concatenate([o.ravel() for o in Omega])).cuda()
    events = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
    for e in events:
        e.record()
    lib().asi_profile_begin(2, (ctypes.c_void_p * 2)(*(e.cuda_event for e in events)), 1)   # ASI_K_EXPAND
    try:
        run.init_factors(act, omega)
    finally:
        seen = lib().asi_profile_end(None)
    assert seen == passes
    assert run.ok()
    S_ref, U_ref = O.asi_cold_start(A.astype(np.float64), [o.astype(np.float64) for o in Omega])
    U = run.factors()
    assert max(O.rel_fro(O.projector(a), O.projector(b)) for a, b in zip(U, U_ref)) <= 1e-4
    assert O.rel_fro(O.sign_align(run.core_np(), U, U_ref)[0], S_ref) <= 1e-4


@pytest.mark.parametrize("dims,ranks", [((33, 128, 20, 20), (6, 5, 7, 5)), ((40, 100, 20, 28), (5, 5, 5, 8))])
def test_bf16_activations_off_sixteen_bytes(dims, ranks):
    """Plans with the tensor-core passes whose activation starts at any element: other kernels on the same number of partials, warm
    and cold, against the oracle."""
    rho = tuple(min(0.7, 0.25 ** (1.0 / max(r - 1, 1))) for r in ranks)
    L = LayerSpec("t", "conv", dims, 6, 3, 1, 1, 1, ranks=ranks)
    st = LayerStream(dims=dims, ranks=ranks, dy_shape=L.dy_shape, seed=sum(dims), rho=rho, bf16=True,
                     gen_ranks=tuple(min(d, max(r + 2, 4)) for d, r in zip(dims, ranks)))
    run = make_runner(L, bf16=True)
    to_device = run.to_device
    U_prev = st.u_prev0()
    A, dY = st.next()
    rng = np.random.default_rng(5)
    n = int(np.prod(dims))
    Omega = [rng.standard_normal((n // d, r)).astype(np.float32) for d, r in zip(dims, ranks)]
    omega = torch.from_numpy(np.concatenate([o.ravel() for o in Omega])).cuda()
    S_ref, U_ref = O.asi_cold_start(A.astype(np.float64), [o.astype(np.float64) for o in Omega])
    for shift in (1, 4):
        def place(x):
            t = to_device(x)
            if x is not A:
                return t
            buf = torch.full((t.numel() + 8,), float("nan"), dtype=t.dtype, device=t.device)
            view = buf[shift:shift + t.numel()].view(t.shape)
            view.copy_(t)
            return view

        run.to_device = place
        err, _ = compare_step(run, L, A, dY, U_prev)
        check(err, TOL_F32, f"{dims} shift={shift}")
        run.init_factors(place(A), omega)
        assert run.ok()
        U = run.factors()
        assert max(O.rel_fro(O.projector(a), O.projector(b)) for a, b in zip(U, U_ref)) <= 1e-4
        assert O.rel_fro(O.sign_align(run.core_np(), U, U_ref)[0], S_ref) <= 1e-4
