"""Roundings of the FP64 2D wave solve in fixed point (csrc/fixed64.cuh) are unbiased: a constant bias b
of the increments moves the level n steps on by b n^2 / 2 quanta (CPU only)."""

import numpy as np

from test_fixed64_host import fx  # noqa: F401


def test_products_round_without_bias(fx):  # noqa: F811
    """The product with a coefficient (53 bits in 64, no multiple of 2^-24): the mean rounding error
    over random levels is 0 within 6 standard deviations of uniform errors."""
    rng = np.random.default_rng(11)
    for scale in (2.0 ** -10, 2.0 ** -4, 0.2, 0.9):
        a = int(rng.uniform(scale, min(1.0, 2 * scale)) * 2.0 ** 53) << 11
        total, count = 0.0, 6000
        for _ in range(count):
            x = int(rng.integers(-2 ** 58, 2 ** 58))
            # d + a x / 2^64 less its value, exactly, in units of 2^-64
            total += float((fx.mac(0, x, a) << 64) - a * x) * 2.0 ** -64
        assert abs(total / count) <= 6 * (1 / 12) ** 0.5 / count ** 0.5, (scale, total / count)


def test_rescaling_rounds_without_bias(fx):  # noqa: F811
    """Shifts by k bits, over whole periods of the low bits: the errors add up to 0 (ties to even)."""
    for k in (1, 2, 3, 5, 8):
        for start in (0, -4096, 123 << 20):
            base = start - start % 2 ** (k + 1)
            total = sum((fx.rescale(base + i, -k) << k) - (base + i) for i in range(2 ** (k + 1)))
            assert total == 0, (k, start)


def test_conversion_rounds_without_bias(fx):  # noqa: F811
    """Doubles to integers: errors of v and -v cancel (halves away from zero)."""
    rng = np.random.default_rng(12)
    for _ in range(2000):
        v = float(rng.normal() * 2.0 ** 40)
        for e in (-5, 0, 3, 20):
            assert fx.from_double(v, e) == -fx.from_double(-v, e)
