"""The exact splittings behind the tensor-core products, checked on the host: three
balanced base-256 digits of the integers of the exact Gram (csrc/gram_int.cu), eight of
those of the FP64 products (csrc/dgemm_tc.cu), three BF16 parts of an FP32 number
(csrc/sgemm_tc.cu), and the bounds that keep their accumulators exact."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

GRAM_TERMS, FP64_TERMS = 5 * 64, 6 * 32  # terms of K between two readings of the accumulators


def gram_digits(q):
    """q + 0x808080 byte by byte, each less 128; the leading byte with its carry."""
    y = (q.astype(np.int64) + 0x808080).astype(np.uint32)
    return [((y >> (8 * (2 - s))) & (0x1FF if s == 0 else 0xFF)).astype(np.int64) - 128 for s in range(3)]


def fp64_digits(X):
    """X + 0x8080808080808080 byte by byte, each less 128."""
    y = X.astype(np.uint64) + np.uint64(0x8080808080808080)
    return [((y >> np.uint64(8 * (7 - s))) & np.uint64(0xFF)).astype(np.int64) - 128 for s in range(8)]


def bf16_exact(d):
    t = torch.from_numpy(np.asarray(d)).to(torch.float32)
    return bool((t.to(torch.bfloat16).to(torch.float32) == t).all())


def test_gram_digits_reproduce_the_integers():
    rng = np.random.default_rng(1)
    q = np.concatenate([rng.integers(-(1 << 23), (1 << 23) + 1, size=20000),
                        [0, 1, -1, 127, 128, -128, -129, 1 << 23, -(1 << 23), (1 << 23) - 1, 1 - (1 << 23), 0x7F7F7F, -0x808080]])
    d = gram_digits(q)
    assert all(x.min() >= -128 and x.max() <= 128 and bf16_exact(x) for x in d)
    assert d[0].max() == 128  # the carry
    np.testing.assert_array_equal(sum(d[s] << (8 * (2 - s)) for s in range(3)), q)


def test_fp64_digits_reproduce_the_integers():
    rng = np.random.default_rng(2)
    X = np.concatenate([rng.integers(-(1 << 62), (1 << 62) + 1, size=20000, dtype=np.int64),
                        np.array([0, 1, -1, 1 << 62, -(1 << 62), (1 << 62) - 512, 0x7F7F7F7F7F7F7F], dtype=np.int64)])
    d = fp64_digits(X)
    assert all(x.min() >= -128 and x.max() <= 128 and bf16_exact(x) for x in d)
    assert np.abs(d[0]).max() <= 64
    np.testing.assert_array_equal(sum((d[s].astype(object) * 256 ** (7 - s)) for s in range(8)), X.astype(object))


def test_sums_stay_below_two_to_24():
    """Largest sums of a level between two readings: three digit products of at most 2^14 each in the Gram; in the FP64
    products s + t + 1 of them at level s + t, those with a leading digit at most 2^13."""
    assert 3 * 128 * 128 * GRAM_TERMS < 1 << 24
    a = np.full((1, GRAM_TERMS), 128.0, dtype=np.float32)
    s = np.float32(0)
    for _ in range(3):
        s = s + (a @ a.T)[0, 0]
    assert s == 3 * 128 * 128 * GRAM_TERMS
    for level in range(6):
        pairs = sum((64 if i == 0 else 128) * (64 if level - i == 0 else 128) for i in range(level + 1))
        assert pairs * FP64_TERMS < 1 << 24


@pytest.mark.parametrize("n2,m,seed", [(4096, 12, 0), (2048, 20, 1), (321, 7, 2), (129, 7, 3)])
def test_gram_from_digits(n2, m, seed):
    """The kernel's sums: FP32 products of the digit rows, levels s + t together, runs of 320 rows, the five levels
    recombined modulo 2^64; G_ij from the rows of real and imaginary parts."""
    rng = np.random.default_rng(seed)
    re = rng.integers(-(1 << 23), (1 << 23) + 1, size=(n2, m))
    im = rng.integers(-(1 << 23), (1 << 23) + 1, size=(n2, m))
    re[:, 0], im[:, 0] = 1 << 23, -(1 << 23)  # the largest magnitudes, with the carry
    rows = np.empty((2 * m, n2), dtype=np.int64)
    rows[0::2], rows[1::2] = re.T, im.T
    d = [x.astype(np.float32) for x in gram_digits(rows)]
    acc = np.zeros((2 * m, 2 * m), dtype=np.uint64)
    for k in range(0, n2, GRAM_TERMS):
        for level in range(5):
            p = np.zeros((2 * m, 2 * m), dtype=np.float32)
            for s in range(3):
                if 0 <= level - s < 3:
                    p += d[s][:, k:k + GRAM_TERMS] @ d[level - s][:, k:k + GRAM_TERMS].T
            assert np.abs(p).max() < 1 << 24
            acc += p.astype(np.int64).astype(np.uint64) << np.uint64(8 * (4 - level))
    S = acc.astype(np.int64)
    a, b = re.astype(np.int64), im.astype(np.int64)
    np.testing.assert_array_equal(S[0::2, 0::2] + S[1::2, 1::2], a.T @ a + b.T @ b)
    np.testing.assert_array_equal(S[0::2, 1::2] - S[1::2, 0::2], a.T @ b - b.T @ a)


def test_bf16_parts_are_exact():
    """x = b0 + b1 + b2 for entries of at least 2^-100, and |b1| <= 2^-8 |b0|, |b2| <= 2^-16 |b0|."""
    rng = np.random.default_rng(3)
    x = torch.from_numpy((rng.standard_normal(100000) * 2.0 ** rng.uniform(-99, 120, 100000)).astype(np.float32))
    x = x[x.abs() >= 2.0 ** -100]
    x = torch.cat([x, torch.tensor([1.0, 1 + 2.0 ** -23, 2 - 2.0 ** -23, 255.5, -1.00390625, 2.0 ** -100])])
    rest, parts = x.clone(), []
    for _ in range(3):
        b = rest.to(torch.bfloat16).to(torch.float32)
        parts.append(b)
        rest = rest - b
    assert bool((rest == 0).all())
    assert bool((parts[1].abs() <= 2.0 ** -8 * parts[0].abs()).all())
    assert bool((parts[2].abs() <= 2.0 ** -16 * parts[0].abs()).all())
