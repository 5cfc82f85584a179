"""The accumulators of the digit products at their limit (csrc/nonlocal_slices.cu): a float32 holds integers exactly up to
2^24, and level 7 takes up to 8 products of two digits in [-128, 127] for each of 128 values of k.

Projector and band are integers built from their digits, all near -128, so that level 7 comes to more than 3/4 of 2^24 with odd
terms.  One unit of it is 2^-68 of such a sum and could not be seen in a float64; so further entries, whose products with a
power of two are exact, cancel all but 62 bits.  What is left is compared with the integer sum of the 36 digit products that
are kept."""
import numpy as np
import pytest

LAT, ECUT, FFT = np.diag([8.0, 8.0, 8.0]), 8.0, (20, 20, 20)
CHUNK = 128   # values of k (two for each plane wave) between two emptyings


def _digits(x):
    """The eight balanced digits of |x| < 2^62, most significant first."""
    out = []
    for _ in range(8):
        d = ((x + 128) & 255) - 128
        out.append(d)
        x = (x - d) >> 8
    assert x == 0
    return out[::-1]


def _kept(a, b):
    """The product of two integers without the digit products of levels 8 to 14."""
    da, db = _digits(a), _digits(b)
    return sum(da[i] * db[j] * 256 ** (14 - i - j) for i in range(8) for j in range(8 - i))


def _rows(npw, seed):
    """Integers a[G], b[G] (0 at G = 0), and the sum over G of twice their kept products."""
    rng = np.random.default_rng(seed)
    a, b = [0] * npw, [0] * npw
    dig = lambda lo, hi, step=1: int(rng.integers(lo // step, hi // step + 1)) * step
    total, used = 0, 0
    for g in range(npw // 2):   # from the first plane wave on, whole chunks
        if used == 3 * CHUNK // 2:
            break
        # 53 significant bits: the last digits of a are 0 and an even one, the last of b is a multiple of 8
        a[g] = sum(d * 256 ** (7 - s) for s, d in enumerate([-63] + [dig(-128, -118) for _ in range(5)] + [dig(-128, -118, 2), 0]))
        b[g] = sum(d * 256 ** (7 - s) for s, d in enumerate([0] + [dig(-128, -118) for _ in range(6)] + [dig(-128, -120, 8)]))
        total += 2 * _kept(a[g], b[g])
        used += 1
    # cancel all but |r| <= 2^61 with products a* 2^61, taken twice
    q = (total + 2 ** 61) >> 62
    r = total - (q << 62)
    g = npw // 2 + 1
    while q:
        x = max(-(2 ** 62 - 512), min(2 ** 62 - 512, q))
        x = int(np.trunc(x / 2.0 ** max(0, abs(x).bit_length() - 53))) << max(0, abs(x).bit_length() - 53)
        a[g], b[g] = -x, 2 ** 61
        assert _kept(a[g], b[g]) == a[g] * b[g]
        q -= x
        g += 1
    assert g < npw and all(int(float(v)) == v for v in a + b)
    return a, b, r, used


def _level7(a, b):
    return sum(x * y for x, y in zip(_digits(a), _digits(b)[::-1]))


def test_rows_reach_the_limit():
    a, b, r, used = _rows(515, 0)
    for c in range(0, used, CHUNK // 2):
        s = 2 * sum(_level7(x, y) for x, y in zip(a[c:c + CHUNK // 2], b[c:c + CHUNK // 2]))
        assert 0.7 * 2 ** 24 < s < 2 ** 24
    assert any(_level7(x, y) % 2 for x, y in zip(a[:used], b[:used]))
    # float32 sums over twice as many values of k would not be exact
    f, exact = np.float32(0.0), 0
    for x, y in zip(a[:used], b[:used]):
        f = np.float32(f + np.float32(2 * _level7(x, y)))
        exact += 2 * _level7(x, y)
    assert abs(r) <= 2 ** 61 and exact > 2 ** 25 and int(f) != exact


@pytest.mark.gpu
@pytest.mark.parametrize("seed", [0, 1])
def test_accumulators_at_their_limit(lib, seed):
    import torch
    from paper_0906_2569_gb300 import binding as B
    m = B.hpsi_gsphere(LAT, ECUT, np.zeros(3))
    npw = len(m)
    a, b, r, _ = _rows(npw, seed)
    P, nb = 17, 2496   # as many tiles of bands as leave one K-split, so that nothing is rounded before the end
    beta = np.zeros((P, npw), dtype=complex)
    beta[1] = np.array([float(x) for x in a]) * (1.0 + 1.0j)
    beta[0, npw // 2] = 1.0
    d = np.zeros((P, P), dtype=complex)
    d[0, 1] = d[1, 0] = 1.0
    ctx = B.hpsi_setup(LAT, ECUT, [np.zeros(3)], FFT, np.zeros(FFT), [beta], d, B.HPSI_FP64,
                       torch.cuda.current_stream().cuda_stream)
    row = torch.from_numpy(np.array([float(x) for x in b]) * (1.0 + 1.0j)).cuda()
    x = row.repeat(nb, 1).contiguous()
    y = torch.full_like(x, float("nan"))
    B.hpsi_apply(ctx, 0, x, y)
    B.hpsi_sync(ctx)
    ctx.close()
    # G = 0: no kinetic term, and <beta_1|psi> through beta_0; r has up to 62 bits: one rounding
    got = y[:, npw // 2].cpu().numpy()
    assert np.all(got.imag == 0.0) and np.all(got.real == got[0].real)
    assert abs(int(got[0].real) - r) <= abs(r) * 2.0 ** -53 + 1


@pytest.mark.gpu
def test_error_is_relative_to_the_largest_entries(lib):
    """A band that is 2^40 at G = 0, where no projector but one has a component: each kept product's operands are rounded at
    2^-62 of their rows' largest entry, and the products left out are below 2^-59 of the rows' largest, for every k."""
    import torch
    from paper_0906_2569_gb300 import binding as B
    m = B.hpsi_gsphere(LAT, ECUT, np.zeros(3))
    npw = len(m)
    rng = np.random.default_rng(5)
    P = 20
    beta = rng.standard_normal((P, npw)) + 1j * rng.standard_normal((P, npw))
    beta[:, npw // 2] = 0.0
    beta[0] = 0.0
    beta[0, npw // 2] = 1.0
    psi = rng.standard_normal((P, npw)) + 1j * rng.standard_normal((P, npw))
    psi[:, npw // 2] = 2.0 ** 40
    d = np.zeros((P, P), dtype=complex)
    d[0, 1:] = d[1:, 0] = 1.0
    ctx = B.hpsi_setup(LAT, ECUT, [np.zeros(3)], FFT, np.zeros(FFT), [beta], d, B.HPSI_FP64,
                       torch.cuda.current_stream().cuda_stream)
    x = torch.from_numpy(psi).cuda()
    y = torch.empty_like(x)
    B.hpsi_apply(ctx, 0, x, y)
    B.hpsi_sync(ctx)
    ctx.close()
    got = y[:, npw // 2].cpu().numpy()   # G = 0: the sum of all projections but beta_0's
    want = (psi @ beta[1:].conj().T).sum(axis=1)   # the numbers at G = 0 drop out: float64 sums of numbers of order 1
    bound = (P - 1) * 2 * npw * (2.0 ** -59 + 2 * 2.0 ** -62) * 2.0 ** 41 * 8.0
    assert np.all(np.abs(got - want) < bound + 1e-10)
