"""The sliced FP64 products (csrc/oz.cu) against double-double arithmetic, tight
enough that two bits fewer in any operand would show, and the row-wise bound that
the header states.

With rows of normal deviates the power-of-two bound of a row is at most 8 of them
(maxima of 4 to 4.5), an element is held to 2^-56 of it (a uniform error of
2^-56 8 / sqrt(3) rms), and both operands' errors over k terms give
sqrt(2) 2^-56 8 / sqrt(3) = 0.8 2^-53 of the result's norm; the result's own
rounding adds at most 0.6 2^-53 (rms), the dropped levels nothing that counts
(k 5 2^-64 64): 1.5 2^-53 in all, 2 2^-53 allowed."""
import pytest

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -53


def _two_prod(a, b):
    """a b = p + e exactly (Dekker 1971; every operation a kernel of its own)."""
    def split(x):
        c = 134217729.0 * x
        hi = c - (c - x)
        return hi, x - hi
    p = a * b
    (ah, al), (bh, bl) = split(a), split(b)
    return p, ((ah * bh - p) + ah * bl + al * bh) + al * bl


def _exact(torch, A, B):
    """B A^T in double-double."""
    h = torch.zeros((B.shape[0], A.shape[0]), dtype=torch.float64, device="cuda")
    l = torch.zeros_like(h)
    for k in range(A.shape[1]):
        p, e = _two_prod(B[:, k, None], A[None, :, k])
        s = h + p
        t = s - h
        l = l + ((h - (s - t)) + (p - t)) + e
        h = s
    return h, l


def _error(ref, C):
    h, l = ref
    return ((C - h) - l).abs()


# one and several tiles with ragged edges, a contraction below a k-block, of
# whole chains (128), of ragged chains and of many
SHAPES = [(1, 1, 1), (5, 70, 31), (128, 64, 128), (130, 66, 129), (257, 130, 1000), (64, 300, 4133)]


@pytest.mark.parametrize("m,n,k", SHAPES)
@pytest.mark.parametrize("splits", [1, 3, 7])
def test_norm_of_the_error(gpu_ctx, m, n, k, splits):
    import torch
    import paper_2502_17963_gb300 as bqc
    g = torch.Generator(device="cuda").manual_seed(m + 7 * n + k)
    A = torch.randn((m, k), generator=g, device="cuda", dtype=torch.float64)
    B = torch.randn((n, k), generator=g, device="cuda", dtype=torch.float64)
    # rows of different sizes: their powers of two scale everything exactly
    A = A * 2.0 ** torch.randint(-40, 40, (m, 1), generator=g, device="cuda")
    B = B * 2.0 ** torch.randint(-40, 40, (n, 1), generator=g, device="cuda")
    C = bqc.gemm_sliced(gpu_ctx, A, B, splits)
    nkb = (k + 31) // 32
    per = 32 * ((nkb + splits - 1) // splits)
    for q in range(splits):
        a, b = A[:, q * per:(q + 1) * per], B[:, q * per:(q + 1) * per]
        if a.shape[1] == 0:
            assert (C[q] == 0).all()
            continue
        err = _error(_exact(torch, a, b), C[q])
        unit = b.norm(dim=1)[:, None] * a.norm(dim=1)[None]  # of each row pair
        scaled = err / unit * a.shape[1] ** 0.5  # as if every result were of size 1
        if m * n >= 300:
            assert scaled.square().mean().sqrt() <= 2 * EPS
        assert scaled.max() <= 16 * EPS  # 6 sigma of it, and rows of a few elements


def test_whole_numbers_are_exact(gpu_ctx):
    """Sums of products of 23-bit integers below 2^53: every digit product that
    is not zero counts."""
    import torch
    import paper_2502_17963_gb300 as bqc
    g = torch.Generator(device="cuda").manual_seed(1)
    A = torch.randint(-2 ** 22, 2 ** 22, (140, 300), generator=g, device="cuda").double()
    B = torch.randint(-2 ** 22, 2 ** 22, (90, 300), generator=g, device="cuda").double()
    assert torch.equal(bqc.gemm_sliced(gpu_ctx, A, B)[0], B @ A.T)


@pytest.mark.parametrize("n", [64, 127, 320])
def test_lower_tiles(gpu_ctx, n):
    import torch
    import paper_2502_17963_gb300 as bqc
    g = torch.Generator(device="cuda").manual_seed(n)
    A = torch.randn((n, 200), generator=g, device="cuda", dtype=torch.float64)
    full, low = (bqc.gemm_sliced(gpu_ctx, A, A, 2, lower) for lower in (False, True))
    j, i = torch.meshgrid(torch.arange(n, device="cuda"), torch.arange(n, device="cuda"),
                          indexing="ij")
    assert torch.equal(full[:, j <= i], low[:, j <= i])


@pytest.mark.parametrize("small", [1e-3, 1e-6, 1e-10])
def test_row_bound(gpu_ctx, small):
    """Rows that are large where the other is small: within k 2^-53 of the rows'
    largest elements (the bound the header gives), which is not relative to the
    element itself."""
    import torch
    import paper_2502_17963_gb300 as bqc
    g = torch.Generator(device="cuda").manual_seed(4)
    k = 4000
    A, B = (torch.randn((64, k), generator=g, device="cuda", dtype=torch.float64) for _ in "AB")
    A[:, : k // 2] *= small
    B[:, k // 2:] *= small
    err = _error(_exact(torch, A, B), bqc.gemm_sliced(gpu_ctx, A, B)[0])
    bound = k * EPS * B.abs().amax(1)[:, None] * A.abs().amax(1)[None]
    assert (err <= bound).all()
