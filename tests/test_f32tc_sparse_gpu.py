"""FP32 products on the tensor cores where few terms of a row are not zero.

Bound for one element, in units u = 2^-24 of |A||B|: the three products left out are at
most 2 u (2^-24 + 2^-24 + 2^-32); the two additions of p0 q0 to a chunk's accumulator are
truncated (2 u each), the ten additions before at 2^-7 of that (0.2 u); every chunk sum and
split partial after the first with a non-zero term is rounded once: 7 + terms + splits.
Products by 0 and by powers of two have one part that is not zero, integers below 2^12 no
third part: their sums below 2^24 are exact."""
import pytest

pytestmark = pytest.mark.gpu
U = 2.0 ** -24
N = 384


@pytest.fixture(scope="module")
def torch():
    import torch as t
    return t


def run(lib, torch, bn, splits, A, B):
    M, K = A.shape
    C = torch.full((M, B.shape[1]), float("nan"), device="cuda")
    lib.f32tc_selftest(bn, splits, "N", "N", M, B.shape[1], K, 1.0, A, K, 0, B, B.shape[1], 0, 0.0, C, B.shape[1], 0)
    torch.cuda.synchronize()
    assert lib.device_status() == 0
    return C


def sparse(torch, terms, signed, seed):
    """N x N, `terms` values in [-1, 1) or [0, 1) at random places of every row."""
    g = torch.Generator("cuda").manual_seed(seed)
    at = torch.rand((N, N), generator=g, device="cuda").topk(terms, 1).indices
    v = torch.rand((N, terms), generator=g, device="cuda")
    return torch.zeros((N, N), device="cuda").scatter_(1, at, v * 2 - 1 if signed else v)


@pytest.mark.parametrize("bn", [64, 128, 256])
@pytest.mark.parametrize("splits", [1, 3])
@pytest.mark.parametrize("terms", [1, 2, 5, 16])
@pytest.mark.parametrize("signed", [True, False])
def test_few_terms_a_row(lib, torch, bn, splits, terms, signed):
    A = sparse(torch, terms, signed, terms)
    B = torch.rand((N, N), generator=torch.Generator("cuda").manual_seed(99), device="cuda") * 2 - 1
    for a, b in ((A, B), (B.t().contiguous(), A.t().contiguous())):
        ref, den = a.double() @ b.double(), a.double().abs() @ b.double().abs()
        assert bool(((run(lib, torch, bn, splits, a, b).double() - ref).abs() <= (7 + terms + splits) * U * den).all())


@pytest.mark.parametrize("bn", [64, 128, 256])
@pytest.mark.parametrize("block", [16, 32, 96])
def test_block_diagonal(lib, torch, bn, block):
    g = torch.Generator("cuda").manual_seed(block)
    A = torch.rand((N, N), generator=g, device="cuda") * 2 - 1
    i = torch.arange(N, device="cuda") // block
    A *= i[:, None] == i[None, :]
    B = torch.rand((N, N), generator=g, device="cuda") * 2 - 1
    ref, den = A.double() @ B.double(), A.double().abs() @ B.double().abs()
    chunks = block // 32 + 2  # that a row's block may lie in
    assert bool(((run(lib, torch, bn, 1, A, B).double() - ref).abs() <= (8 + chunks) * U * den).all())


@pytest.mark.parametrize("bn", [64, 128, 256])
@pytest.mark.parametrize("splits", [1, 3])
def test_permutations_and_powers_of_two_bit_for_bit(lib, torch, bn, splits):
    g = torch.Generator("cuda").manual_seed(5)
    X = torch.randn((N, N), generator=g, device="cuda")
    X[0, :] = 1 + 2.0 ** -23
    X[1, :] = 2 - 2.0 ** -23
    X[2, ::2] = -(2.0 ** -100)
    perm = torch.randperm(N, generator=g, device="cuda")
    P = torch.zeros((N, N), device="cuda")
    P[torch.arange(N, device="cuda"), perm] = 1
    assert torch.equal(run(lib, torch, bn, splits, P, X), X[perm])
    assert torch.equal(run(lib, torch, bn, splits, X, P.t().contiguous()), X[:, perm])
    scale = 2.0 ** torch.randint(-20, 20, (N,), generator=g, device="cuda").float()
    assert torch.equal(run(lib, torch, bn, splits, P * scale[:, None], X), X[perm] * scale[:, None])
    assert torch.equal(run(lib, torch, bn, splits, -P, X), -X[perm])


@pytest.mark.parametrize("bn", [64, 128, 256])
def test_products_of_12_bit_integers(lib, torch, bn):
    g = torch.Generator("cuda").manual_seed(6)
    d = torch.randint(-4095, 4096, (N,), generator=g, device="cuda").float()
    X = torch.randint(-4095, 4096, (N, N), generator=g, device="cuda").float()
    assert torch.equal(run(lib, torch, bn, 1, torch.diag(d), X), d[:, None] * X)
