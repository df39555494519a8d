"""The two-part TF32 split of the persistent kernel's tile updates.

x = h + l with h the nearest TF32 value (10 fraction bits) and l exact; the
tensor core reads l's leading 11 significant bits.  Three products (h h, h l,
l h) then miss a product a b by at most 2^-22 + 2 2^-22 of |a b|: l l is at
most 2^-11 x 2^-11, and dropping l's last bit loses at most 2^-22 of each
factor.  A K-long sum stays within that of the sum of magnitudes, where TF32
alone would not.
"""
import numpy as np


def _tf32(x, up):
    b = np.asarray(x, np.float32).view(np.uint32)
    return ((b + np.uint32(0x1000 if up else 0)) & np.uint32(0xFFFFE000)).view(np.float32)


def _split(x):
    h = _tf32(x, True)
    l = (x - h).astype(np.float32)
    assert np.array_equal(h.astype(np.float64) + l, x.astype(np.float64))  # exact
    return h, _tf32(l, False)


def test_three_products_keep_fp32_accuracy():
    rng = np.random.default_rng(0)
    a = (rng.normal(size=(4096, 104)) * 10.0 ** rng.uniform(-3, 3, size=(4096, 1))).astype(np.float32)
    b = rng.normal(size=(4096, 104)).astype(np.float32)
    (ah, al), (bh, bl) = _split(a), _split(b)
    f = np.float64
    got = (ah.astype(f) * bh + ah.astype(f) * bl + al.astype(f) * bh).sum(1)
    ref = (a.astype(f) * b).sum(1)
    mag = np.abs(a.astype(f) * b).sum(1)
    assert (np.abs(got - ref) / mag).max() <= 3 * 2.0 ** -22
    one = (ah.astype(f) * bh).sum(1)
    assert (np.abs(one - ref) / mag).max() > 2.0 ** -16  # the control: one product alone
