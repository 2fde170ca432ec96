"""Modes of 2^31 columns: tensors of more elements than 32 bits count, against torch in fp64."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _mode_product(A, m, V):
    """P = A_m V for one column V [b_m], in fp64 over pieces of the tensor."""
    a = A.shape[m]
    X = A.reshape(A.shape[:m].numel(), a, -1)
    V = V.view(X.shape[0], X.shape[2])
    P = torch.zeros(a, dtype=torch.float64, device=A.device)
    for o, i, x in _pieces(X):
        P += torch.einsum("oai,oi->a", x, V[o, i].double())
    return P


def _columns(A, m, u):
    """V = A_m^T u as fp32 [b_m]."""
    X = A.reshape(A.shape[:m].numel(), A.shape[m], -1)
    V = torch.empty(X.shape[0], X.shape[2], device=A.device)
    for o, i, x in _pieces(X):
        V[o, i] = torch.einsum("oai,a->oi", x, u.double()).float()
    return V.view(-1)


def _pieces(X, most=1 << 29):
    O, a, I = X.shape
    step_i = min(I, most // a)
    step_o = max(1, most // (a * step_i))
    for o in range(0, O, step_o):
        for i in range(0, I, step_i):
            so, si = slice(o, o + step_o), slice(i, i + step_i)
            yield so, si, X[so, :, si].double()


@pytest.mark.parametrize("dims,generic", [((2, 2, 32768, 32768), False), ((2, 2, 32768, 32768), True)])
def test_modes_of_2_to_the_31_columns(dims, generic):
    """Cold start and one warm step at ranks 1 on 2^32 bf16 values: modes 1 and 2 have 2^31 columns, in one slab and in
    two of 2^30.  At rank 1, U_m = P_m / |P_m|; an fp32 sum of 2^31 products in splits of a few million is good to
    about 1e-4 of the sum's random walk."""
    if torch.cuda.get_device_properties(0).total_memory < 100 * 2 ** 30:
        pytest.skip("needs 60 GB of device memory")
    from paper_2505_05086_b200.runner import LayerRunner
    gen = torch.Generator(device="cuda").manual_seed(31)
    A = torch.empty(dims, dtype=torch.bfloat16, device="cuda")
    flat = A.view(-1)
    for i in range(0, flat.numel(), 1 << 28):
        flat[i:i + (1 << 28)] = torch.randn(1 << 28, generator=gen, device="cuda").bfloat16()
    # a common part that grows towards the end of every mode, so that no columns may be missing
    A[:, 1, 20000:, :] += 1.0
    A[1, :, :, 30000:] += 2.0
    run = LayerRunner("conv", dims, (1, 1, 1, 1), 1, bf16=True, generic_only=generic)
    b = [A.numel() // d for d in dims]
    omega = torch.randn(sum(b), generator=gen, device="cuda") + 0.25
    run.init_factors(A, omega)
    assert run.ok()
    cold = [torch.from_numpy(u[:, 0]).cuda().double() for u in run.factors()]
    at = 0
    for m, n in enumerate(b):
        P = _mode_product(A, m, omega[at:at + n])
        at += n
        want = P / P.norm()
        assert float((cold[m] - want).norm()) < 1e-4, m
    del omega
    run.compress(A)
    assert run.ok()
    warm = [torch.from_numpy(u[:, 0]).cuda().double() for u in run.factors()]
    for m in range(4):
        P = _mode_product(A, m, _columns(A, m, cold[m]))
        want = P / P.norm()
        assert float((warm[m] - want).norm()) < 1e-4, m
    total = 0.0
    for x in range(2):
        for y in range(2):
            v = torch.zeros(dims[2], dtype=torch.float64, device="cuda")
            for h in range(0, dims[2], 4096):
                v[h:h + 4096] = A[x, y, h:h + 4096].double() @ warm[3]
            total += float(warm[0][x] * warm[1][y] * (v @ warm[2]))
    assert abs(float(run.core[0]) - total) < 1e-4 * abs(total)
