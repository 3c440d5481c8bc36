"""The quotient from a rounded reciprocal that the small CG's scalars use (q = a y,
then one correction by the remainder's quotient) rounds as the division does:
every pair of significands of 5 to 9 bits, in integers, with the remainder
rounded where it does not fit (the CUDA code is compared with CUDA's division in
test_gpu_arith.py)."""
import pytest


def rounded(m, e, p):
    """m 2^e rounded to p bits, to nearest, ties to even: (significand, exponent)."""
    sign, m = (-1 if m < 0 else 1), abs(m)
    s = max(0, m.bit_length() - p)
    q, r = m >> s, m & ((1 << s) - 1)
    if s and (2 * r > 1 << s or (2 * r == 1 << s and q & 1)):
        q += 1
    return sign * q, e + s


def divided(a, b, p):
    """a / b of two p-bit integers, rounded to p bits."""
    e = -p if a < b else 1 - p
    q, r = divmod(a << -e, b)
    if 2 * r > b or (2 * r == b and q & 1):
        q += 1
    return q, e


def add(m, e, n, f):
    g = min(e, f)
    return (m << (e - g)) + (n << (f - g)), g


@pytest.mark.parametrize("p", [5, 6, 7, 8, 9])
def test_one_correction_rounds_correctly(p):
    inexact = 0
    for b in range(1 << (p - 1), 1 << p):
        y, ye = divided(1 << (p - 1), b, p)
        ye -= p - 1  # 1 / b
        for a in range(1 << (p - 1), 1 << p):
            q, qe = rounded(a * y, ye, p)
            m, e = add(a, 0, -b * q, qe)
            r, re = rounded(m, e, p)
            inexact += r << (re - e) != m
            m, e = add(q, qe, r * y, re + ye)
            got, ge = rounded(m, e, p)
            want, we = divided(a, b, p)
            assert add(got, ge, -want, we)[0] == 0, (a, b)
    assert inexact > 0  # the case that needs more than the usual argument occurs
