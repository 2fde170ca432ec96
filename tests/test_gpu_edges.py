"""The kernels of the warm step at the edges of their tiles, element by element against the fp64 oracle."""
import pytest
import torch

from asi_inputs.configs import LayerSpec
from asi_inputs.generator import LayerStream
from tests.gpu_util import TOL_F32, check, compare_step, make_runner

pytestmark = pytest.mark.gpu


def _rho(r):
    return min(0.7, 0.25 ** (1.0 / max(r - 1, 1)))


def _two_steps(L, bf16, fused=None, rho=None, tol=TOL_F32):
    st = LayerStream(dims=L.dims, ranks=L.ranks, dy_shape=L.dy_shape, seed=sum(L.dims) + L.cout, bf16=bf16,
                     rho=rho or tuple(_rho(r) for r in L.ranks),
                     gen_ranks=tuple(min(d, max(2 * r, r + 2, 4)) for d, r in zip(L.dims, L.ranks)))
    run = make_runner(L, bf16=bf16)
    if fused is not None:
        assert (run.plan.launch_count(0) == 3) == fused
    U_prev = st.u_prev0()
    for _ in range(2):
        A, dY = st.next()
        err, U_prev = compare_step(run, L, A, dY, U_prev)
        check(err, tol, f"{L.dims} {L.ranks} bf16={bf16}")


# Fused small maps of any shape and any batch: (dims, ranks, cout, k, stride, pad, groups)
ANY_MAP = [
    ((3, 9, 6, 11), (2, 4, 3, 4), 7, 3, 1, 1, 1),          # fewer samples than a CTA has warps
    ((13, 33, 7, 7), (4, 4, 4, 3), 12, 3, 1, 1, 1),        # batch not a multiple of eight, C H W odd
    ((17, 40, 16, 16), (3, 8, 5, 8), 8, 3, 1, 1, 2),       # 256 positions, several CTAs per sample
    ((70, 21, 8, 32), (4, 5, 4, 6), 9, 1, 1, 0, 1),        # a row of 32 lanes, batch above one warp's share
    ((10, 130, 6, 6), (4, 4, 4, 4), 20, 3, 2, 1, 1),       # channels beyond one tile
    ((9, 6, 1, 5), (3, 4, 1, 2), 4, 1, 1, 0, 1),           # one row
    ((64, 512, 7, 7), (4, 4, 4, 4), 8, 3, 1, 1, 1),        # one staging block for four rounds of output channels
]


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("case", ANY_MAP)
def test_fused_maps_of_any_shape_and_batch(case, bf16):
    dims, ranks, cout, k, s, p, g = case
    _two_steps(LayerSpec("t", "conv", dims, cout, k, s, p, g, ranks=ranks), bf16, fused=True)


# Planes and strided fibers streamed by warps: odd and even widths, one plane a tile and many, rows or columns shared
# by 2..8 lanes, the largest map; channel modes around 32, 64 and 128 rows; rows that start at any element
STREAMED = [
    ((4, 33, 17, 19), (3, 4, 4, 4)),
    ((3, 64, 9, 50), (3, 5, 5, 6)),                        # few rows: eight lanes a row
    ((2, 65, 50, 9), (2, 6, 6, 5)),                        # few columns: lanes share a pair
    ((2, 31, 33, 33), (2, 4, 4, 4)),                       # two rows a lane, one plane a tile
    ((3, 128, 27, 27), (3, 8, 5, 5)),                      # the longest fiber; odd planes
    ((2, 12, 64, 64), (2, 8, 8, 8)),                       # the largest map, ranks 8
    ((40, 7, 20, 24), (8, 4, 4, 4)),                       # vector copies along the batch, rank 8
    ((5, 12, 60, 36), (3, 3, 3, 3)),                       # planes of unequal sides, aligned rows
    ((129, 5, 18, 18), (4, 3, 4, 4)),                      # a batch one past the fiber kernels
]


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("dims,ranks", STREAMED)
def test_streamed_planes_and_fibers(dims, ranks, bf16):
    _two_steps(LayerSpec("t", "conv", dims, 10, 3, 2, 1, 1, ranks=ranks), bf16, fused=False)


def test_a_stride_two_layer_with_a_large_product_on_the_streamed_fibers():
    """The first core product and Z1 of a layer of a million values, rows of an odd length."""
    _two_steps(LayerSpec("t", "conv", (50, 40, 27, 27), 45, 3, 1, 1, 1, ranks=(5, 4, 4, 4)), False, fused=False)


# Grouped products and Orthogonalize of token layers: ranks on both sides of 8, 16, 32 and 64, ragged token counts and
# features, two modes and three
GROUPED = [
    ((5, 33, 31), (1, 9, 17)),
    ((9, 100, 70), (9, 16, 33)),
    ((3, 129, 257), (2, 8, 32)),
    ((130, 70), (65, 40)),
    ((140, 127), (17, 24)),
    ((300, 96), (32, 64)),
]


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("dims,ranks", GROUPED)
def test_grouped_products_at_the_edges(dims, ranks, bf16):
    rho = tuple(0.25 ** (1.0 / max(r, 4)) for r in ranks)
    _two_steps(LayerSpec("t", "linear", dims, 37, ranks=ranks), bf16, rho=rho, tol=dict(TOL_F32, proj=1e-3, dw=1e-3))


@pytest.mark.parametrize("dims", [(23, 40, 1664), (37, 72, 1088)])
def test_tensor_core_products_with_several_tiles_a_cta(dims):
    """299 and 333 tiles of the token products: two a CTA, the last CTA one; the second token count has a ragged chunk."""
    ranks = (3, 16, 16)
    _two_steps(LayerSpec("t", "linear", dims, 1600, ranks=ranks), True, rho=(0.6, 0.93, 0.93),
               tol=dict(TOL_F32, proj=1e-3))


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("dims", [(128, 1280), (70, 1290), (33, 390)])
def test_long_contractions_of_few_tiles(dims, bf16):
    """Tiles shared by clusters of 8 and 2 CTAs, the last ones with an empty or a ragged share of the contraction."""
    ranks = (12, 14)
    _two_steps(LayerSpec("t", "linear", dims, 40, ranks=ranks), bf16, rho=(0.9, 0.9), tol=dict(TOL_F32, proj=1e-3))


# Tensors that start at any element: (dims, ranks, cout, kernel, act shifted too).  Square maps with whole tiles, maps
# with their samples over clusters, columns that come in whole groups of four and not, a weight gradient behind a large map
SHIFTED = [
    ((8, 32, 16, 16), (4, 8, 8, 8), 32, 3, True),
    ((16, 16, 7, 7), (3, 4, 4, 4), 12, 3, True),
    ((8, 12, 14, 14), (3, 4, 4, 4), 8, 1, True),
    ((136, 20, 7, 7), (4, 4, 4, 4), 12, 3, True),
    ((6, 3, 4, 5), (4, 3, 4, 4), 8, 3, True),
    ((13, 33, 7, 7), (4, 4, 4, 3), 12, 3, True),
    ((17, 40, 16, 16), (3, 8, 5, 8), 8, 3, True),
    ((11, 64, 14, 14), (4, 4, 4, 4), 16, 3, True),
    ((55, 9, 28, 28), (5, 2, 3, 4), 257, 3, False),
    ((9, 12, 20, 24), (8, 5, 5, 5), 16, 3, False),
    ((9, 13, 19, 23), (8, 5, 5, 5), 16, 3, True),
]


@pytest.mark.parametrize("shift", [1, 2, 3])
@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("case", SHIFTED)
def test_tensors_that_start_at_any_element(case, bf16, shift):
    dims, ranks, cout, k, act_too = case
    L = LayerSpec("t", "conv", dims, cout, k, 1, k // 2, 1, ranks=ranks)
    st = LayerStream(dims=L.dims, ranks=L.ranks, dy_shape=L.dy_shape, seed=sum(L.dims) + L.cout, bf16=bf16,
                     rho=tuple(_rho(r) for r in L.ranks),
                     gen_ranks=tuple(min(d, max(2 * r, r + 2, 4)) for d, r in zip(L.dims, L.ranks)))
    run = make_runner(L, bf16=bf16)
    to_device = run.to_device

    def shifted(x):
        t = to_device(x)
        if x.shape == tuple(L.dims) and not act_too:
            return t
        buf = torch.full((t.numel() + 8,), float("nan"), dtype=t.dtype, device=t.device)
        view = buf[shift:shift + t.numel()].view(t.shape)
        view.copy_(t)
        assert view.data_ptr() % 16 == shift * t.element_size()
        return view

    run.to_device = shifted
    A, dY = st.next()
    err, _ = compare_step(run, L, A, dY, st.u_prev0())
    check(err, TOL_F32, f"{dims} {ranks} bf16={bf16} shift={shift}")
    with pytest.raises(Exception, match="invalid argument"):      # half an element is refused, not read
        run.plan.wgrad(run.core.data_ptr(), run.U[run.cur].data_ptr(), to_device(dY).data_ptr() + 1, run.dW.data_ptr(),
                       run.ws_w.data_ptr(), run.ws_w.numel())


@pytest.mark.parametrize("dims,ranks,split", [((24, 384), (5, 5), False), ((24, 385), (5, 5), True), ((520, 40), (8, 8), True),
                                              ((6, 20, 1300), (3, 8, 8), True), ((3, 512, 18, 18), (3, 8, 4, 4), False),
                                              ((3, 513, 18, 18), (3, 4, 4, 4), True)])
def test_rows_of_the_factors_on_both_sides_of_the_factoring_cta(dims, ranks, split):
    """Ranks up to eight: 384 rows (conv layers: 512) are solved by the CTA that factors the mode, more in a launch of their own."""
    def layer(d):
        return LayerSpec("t", "conv", d, 6, 3, 1, 1, 1, ranks=ranks) if len(d) == 4 else LayerSpec("t", "linear", d, 37, ranks=ranks)

    run, short = make_runner(layer(dims)), make_runner(layer(tuple(min(d, 512 if len(dims) == 4 else 384) for d in dims)))
    assert run.plan.launch_count(0) == short.plan.launch_count(0) + split
    _two_steps(layer(dims), False)


@pytest.mark.parametrize("rank", [1, 4, 11, 12, 13])
@pytest.mark.parametrize("cout", [64, 67])
def test_weight_gradients_of_short_sums(rank, cout):
    """Both forms of the last product of a linear layer, whole tiles and ragged ones, ranks that are whole groups of four and not."""
    _two_steps(LayerSpec("t", "linear", (48, 131), cout, ranks=(rank, rank)), False, rho=(0.9, 0.9), tol=dict(TOL_F32, proj=1e-3))
