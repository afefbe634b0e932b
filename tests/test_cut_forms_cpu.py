"""Forms of the selection's steps that must equal their plain ones, restated in FP32 numpy:
the packed partner masks, the azimuth wrap of the 4th-hit metric, the order that replaces the
address in its tie rule, and the numbering of the e+ pairs."""
import numpy as np
import pytest

from paper_2206_11535_gb300 import gen

F = np.float32


@pytest.mark.parametrize("n", [1, 3, 4, 31, 32])
def test_sign_of_the_difference_is_the_comparison(n):
    """bit q of the mask: product >= c, taken as the sign of product - c, last hit first."""
    r = np.random.default_rng(n)
    c = F(r.uniform(100.0, 800.0))
    near = np.nextafter(c, r.choice(np.array([0.0, 1e9], F), n)).astype(F)
    dot = np.where(r.random(n) < 0.3, c, np.where(r.random(n) < 0.5, near, r.uniform(-900, 900, n))).astype(F)
    m = 0
    padded = np.concatenate([dot, r.uniform(-900, 900, -n % 4).astype(F)])
    for q in range(padded.size - 1, -1, -1):
        m = ((m << 1) | int(np.signbit(F(padded[q] + F(-c))))) & 0xFFFFFFFF
    below = (1 << n) - 1
    assert (~m & below) == sum(1 << q for q in range(n) if dot[q] >= c)


def test_azimuth_wrap_takes_the_shorter_way():
    two_pi = F(2 * np.pi)
    r = np.random.default_rng(5)
    d = np.concatenate([r.uniform(-6.28, 6.28, 200_000), r.uniform(-1e-3, 1e-3, 1000), [0.0]]).astype(F)
    a = np.abs(d)
    got = np.minimum(a, (two_pi - a).astype(F))
    # the difference less the nearest multiple of 2 pi, rounded once
    k = np.rint((d * F(1 / (2 * np.pi))).astype(F)).astype(np.float64)
    want = np.abs((d.astype(np.float64) - k * np.float64(two_pi)).astype(F))
    clear = np.abs(a - F(np.pi)) > 1e-5  # at a half turn both ways are equally long
    assert (got[clear] == want[clear]).all()
    assert np.allclose(got, want, atol=2e-6)


@pytest.mark.parametrize("n_cols,n_rows,pitch", [(None, None, None), (256, 8192, 0.02), (1, 1, 0.5)])
def test_coordinates_order_a_layer_as_addresses_do(n_cols, n_rows, pitch):
    """phi grows with (ladder, column) and z with the row, strictly, as FP32 values."""
    g = gen.load_config()["geometry"]
    for L in range(4):
        nl = g["n_ladders"][L] if n_cols is None else 32
        nt = nl * (g["n_cols"][L] if n_cols is None else n_cols)
        phi = ((np.arange(nt) + 0.5) * 2.0 * np.pi / nt).astype(F)
        z = (-g["half_len_mm"][L] + (np.arange(g["n_rows"][L] if n_rows is None else n_rows) + 0.5)
             * (g["pitch_mm"] if pitch is None else pitch)).astype(F)
        assert (np.diff(phi) > 0).all() and (np.diff(z) > 0).all()


def test_pair_numbering_is_exact_with_one_correction():
    n = 128
    pr = np.arange(n * (n - 1) // 2)
    for ulps in (-1, 0, 1):  # the root may be off by a rounding
        root = np.sqrt((1 + 8 * pr).astype(F)).astype(F)
        for _ in range(abs(ulps)):
            root = np.nextafter(root, F(ulps * 1e9))
        b = ((F(1) + root).astype(F) * F(0.5)).astype(np.int64)
        b = np.where(b * (b - 1) // 2 > pr, b - 1, b)
        b = np.where((b + 1) * b // 2 <= pr, b + 1, b)
        a = pr - b * (b - 1) // 2
        want = [(i, j) for j in range(n) for i in range(j)]
        assert list(zip(a.tolist(), b.tolist())) == want
