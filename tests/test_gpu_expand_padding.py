"""Columns k .. ld - 1 of an expansion are those of Z (zero without Z), also where the padding is
wider than the column blocks and chunks that the kernels write."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("tensor_cores", [True, False])
@pytest.mark.parametrize("with_z", [True, False])
@pytest.mark.parametrize("k,ld", [(8, 64), (8, 68), (64, 72), (65, 260), (100, 640), (3, 1200)])
def test_padding(gpu_bmg, dtype, tensor_cores, with_z, k, ld):
    g = torch.Generator(device="cuda").manual_seed(ld)
    n = 300
    X, Z = (torch.randn((n, ld), dtype=dtype, device="cuda", generator=g) for _ in range(2))
    Y = torch.randn((k, k), dtype=torch.float64, device="cuda", generator=g)
    U = torch.full_like(X, float("nan"))
    if not tensor_cores and k * ld * X.element_size() > 227 * 1024:
        pytest.skip("the coefficients do not fit in shared memory: refused")
    gpu_bmg.expand(Z if with_z else None, X, Y, k, U, tensor_cores)
    assert torch.equal(U[:, k:], Z[:, k:] if with_z else torch.zeros_like(Z[:, k:]))
    ref = X[:, :k].double() @ Y + (Z[:, :k].double() if with_z else 0.0)
    tol = 1e-12 if dtype == torch.float64 else 1e-4       # far above the roundings of 100 products
    assert (U[:, :k].double() - ref).abs().max().item() <= tol
