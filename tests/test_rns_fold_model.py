"""The running sum of residues in the tensor-core product's epilogue (FP32,
one addend of at most p / 2 + 1 <= 256 per 256 k): exact only while it stays
within 2^24, so it is reduced mod p every 32768 addends.  CPU model at the
worst case, addends of one sign (a product of constant matrices)."""
import numpy as np
import pytest

P, FOLD = 511, 32768


def _mod(v, p):
    """v - round(v / p) p in FP32, as the kernel forms it."""
    inv = np.float32(1.0) / np.float32(p)
    magic = np.float32(12582912.0)
    q = np.float32(np.float32(np.float64(v) * np.float64(inv) + np.float64(magic)) - magic)
    return np.float32(np.float64(v) - np.float64(q) * p)


def _run(addend, count, fold):
    acc, left, done = np.float32(0), fold, 0
    while done < count:
        step = min(left, count - done)
        # FP32 additions of one value, stepwise only where they can round
        exact = float(acc) + addend * step
        if abs(exact) <= 2 ** 24:
            acc = np.float32(exact)
        else:
            for _ in range(step):
                acc = np.float32(acc + np.float32(addend))
        done += step
        left -= step
        if left == 0:
            left, acc = fold, _mod(acc, P)
    return acc


@pytest.mark.parametrize("addend", [251, -255, 1])
@pytest.mark.parametrize("count", [1, FOLD, FOLD + 1, 70001, 200003])
def test_folded_sum_is_exact(addend, count):
    assert (int(_run(addend, count, FOLD)) - addend * count) % P == 0
    assert abs(float(_run(addend, FOLD, FOLD + 1))) <= 2 ** 24


def test_without_the_fold_long_sums_round():
    got = _run(251, 70001, 10 ** 9)
    assert (int(got) - 251 * 70001) % P != 0
