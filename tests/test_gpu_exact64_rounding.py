"""FP64 quotients and roots of exact64.cuh where they are hardest to round: operands whose exact
quotient or root lies as near to the middle between two doubles as any can, divisors with a mantissa
of ones (the one for which a correctly rounded reciprocal is not enough), zeros of both signs.  The
library's entry points give the IEEE results, bit for bit: m / rho of cons_to_prim, and the sound
speed sqrt(gamma p / rho) behind cfl_dt."""
import numpy as np
import pytest

from paper_1204_4779_gb300 import hydro

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
F64 = torch.float64


def _quotients(a, b):
    """a / b as the momentum and density of a 1D state (the energy keeps the pressure positive)."""
    U = np.stack([b, a, a * a / b + b])
    return hydro.cons_to_prim(torch.from_numpy(U).cuda(), 1.4)[1].cpu().numpy()


def _same_bits(x, y):
    return np.array_equal(x.view(np.int64), y.view(np.int64))


def _near_midpoints(B, ks):
    """Mantissas A in [2^52, B) with A 2^54 = B (2 M + 1) + k: A / B is |k| / (2 B) units of the
    last place from the middle of two doubles."""
    inv = pow(pow(2, 54, B), -1, B)
    out = [k * inv % B for k in ks]
    return [A for A in out if A >= 1 << 52]


@pytest.mark.parametrize("log_j", [0, 3, 9, 20, 26, 29, 33, 36, 38, 41, 47, 51])
def test_quotients_next_to_midpoints(log_j):
    """Divisors 2^53 - j, j odd around 2^log_j."""
    rng = np.random.default_rng(log_j)
    ks = [s * (2 * i + 1) for i in range(4) for s in (1, -1)]
    a, b = [], []
    for _ in range(1 if log_j == 0 else 400):
        B = (1 << 53) - (int(rng.integers(1 << log_j, 2 << log_j)) | 1)
        for A in _near_midpoints(B, ks):
            a.append(float(A))
            b.append(float(B))
    a, b = np.array(a), np.array(b)
    for sign, ea, eb in ((1, 0, 0), (-1, -53, -52), (1, 100, -101), (-1, -200, 150)):
        x, y = sign * np.ldexp(a, ea), np.ldexp(b, eb)
        assert _same_bits(_quotients(x, y), x / y), (log_j, ea, eb)


def _reciprocals_next_to_midpoints(rng, log_j, count):
    """Divisors B = 2^53 - j, j around 2^log_j, with 1 / B less than 2^-17 units of the last place
    from the middle of two doubles: the part of 2^105 / B after the point moves by about
    j 2^-52 from one odd j to the next."""
    out = []
    while len(out) < count:
        j = 2 * int(rng.integers(1 << (log_j - 1), 1 << log_j)) + 1
        side = 0.5 + rng.uniform(-1.0, 1.0) * 2.0 ** -17
        for _ in range(4):
            B = (1 << 53) - j
            part = ((1 << 105) % B) / B
            j += 2 * round((side - part) / (j * 2.0 ** -52))
        B = (1 << 53) - j
        if 1 << log_j <= j < 4 << log_j and abs(((1 << 105) % B) / B - 0.5) < 2.0 ** -17:
            out.append(B)
    return out


@pytest.mark.parametrize("log_j", [27, 28, 29, 30, 31, 32, 33, 34])
def test_divisors_with_reciprocals_next_to_midpoints(log_j):
    """An approximate reciprocal may round the wrong way there, and a quotient by it that lies next
    to a midpoint itself with it (only where the divisor's leading mantissa bits are ones)."""
    rng = np.random.default_rng(log_j)
    a, b = [], []
    for B in _reciprocals_next_to_midpoints(rng, log_j, 1000):
        for A in _near_midpoints(B, [1, -1]):
            a.append(float(A))
            b.append(float(B))
    a, b = np.array(a), np.array(b)
    assert len(a) >= 500
    assert _same_bits(_quotients(a, b), a / b)


def test_divisors_of_ones():
    """rho just below a power of two, the momentum a power of two or close to one."""
    a = np.array([1.0 + i * 2.0 ** -52 for i in range(64)] + [1.0 - i * 2.0 ** -53 for i in range(64)])
    for e in (-30, -1, 0, 1, 40):
        b = np.full_like(a, np.ldexp(1.0 - 2.0 ** -53, e))
        assert _same_bits(_quotients(a, b), a / b), e


def test_random_quotients():
    rng = np.random.default_rng(1)
    n = 1 << 20
    b = np.ldexp(rng.uniform(1.0, 2.0, n), rng.integers(-60, 60, n))
    b[: n // 4] = np.ldexp(1.0 - rng.integers(1, 1 << 14, n // 4) * 2.0 ** -53, rng.integers(-3, 3, n // 4))
    a = rng.choice([-1.0, 1.0], n) * np.ldexp(rng.uniform(1.0, 2.0, n), rng.integers(-60, 60, n))
    a[::3] = np.ldexp(1.0, rng.integers(-3, 3, len(a[::3])))
    assert _same_bits(_quotients(a, b), a / b)


def test_zeros_keep_their_sign():
    a = np.array([0.0, -0.0, 0.0, -0.0])
    b = np.array([1.0, 1.0, 0.3, 7.5])
    assert _same_bits(_quotients(a, b), a / b)


def _roots_next_to_midpoints(bits, count):
    """Doubles a = A 2^-52 in [1, 2) (bits 54) or 2 A 2^-52 in [2, 4) (bits 55) with
    A 2^bits = W^2 - c, W odd: sqrt is about |c| 2^-56 units of the last place from the middle."""
    out = []
    for i in range(-count, count):
        c = 1 + 8 * i
        r = 1
        for n in range(3, bits):  # r^2 = c modulo 2^(n + 1)
            if (r * r - c) % (2 << n):
                r += 1 << (n - 1)
        for W in (r, -r, r + (1 << (bits - 1)), -r + (1 << (bits - 1))):
            W %= 1 << bits
            for V in (W, W + (1 << bits)):
                A, rest = divmod(V * V - c, 1 << bits)
                if rest == 0 and V >= 1 << 53 and (1 << 52) <= A < (1 << 53) and V < (1 << 54):
                    out.append(A * 2.0 ** -52 * (2.0 if bits == 55 else 1.0))
    return out


# dt = cfl dr / c tells neighbouring sound speeds c apart where c^2 / 2 <= cfl < c
@pytest.mark.parametrize("bits,cfl,least,most", [(54, 1.0, 1.0, 1.41), (55, 1.41, 1.415, 1.67)])
def test_roots_next_to_midpoints(bits, cfl, least, most):
    """gamma = 2, rho = 1, v = 0: c = sqrt(2 p), and p = E."""
    roots = [a for a in _roots_next_to_midpoints(bits, 300) if least <= a ** 0.5 <= most]
    assert len(roots) > 100
    S = hydro.Solver((64,), 2.0, dtype=F64, cfl=cfl)
    U = torch.zeros((3, 64), dtype=F64, device="cuda")
    U[0] = 1.0
    wrong = []
    for a in roots:
        U[2] = 0.5 * a
        if S.cfl_dt(U) != cfl / (np.sqrt(np.float64(a)) / (1.0 / 64.0)):
            wrong.append(a)
    assert not wrong, (len(wrong), len(roots), wrong[:4])


def test_roots_just_below_powers_of_four():
    """sqrt(1 - 2^-53) lies just below the middle of 1 - 2^-53 and 1."""
    S = hydro.Solver((64,), 2.0, dtype=F64, cfl=1.0)
    U = torch.zeros((3, 64), dtype=F64, device="cuda")
    U[0] = 1.0
    for i in range(1, 40):
        a = 1.0 - i * 2.0 ** -53
        for b in (4.0 * a, a, 0.25 * a):
            U[2] = 0.5 * b
            assert S.cfl_dt(U) == 1.0 / (np.sqrt(np.float64(b)) / (1.0 / 64.0)), (i, b)
