"""Shared helpers of the GPU parity tests (metrics and host<->device plumbing only)."""
import numpy as np


def rel_fro(got, want):
    got = np.asarray(got, np.float64)
    want = np.asarray(want, np.float64)
    d = np.linalg.norm((got - want).ravel())
    n = np.linalg.norm(want.ravel())
    return d / n if n > 0 else d


def same_bits(a, b):
    a = np.ascontiguousarray(a, np.float32)
    b = np.ascontiguousarray(b, np.float32)
    return a.shape == b.shape and np.array_equal(a.view(np.uint32), b.view(np.uint32))


def same_classes(got, want, rel=1e-4):
    """NaN where NaN is expected, the same infinities, and finite values as close as `rel` of the largest."""
    got, want = np.asarray(got, np.float64), np.asarray(want, np.float64)
    finite = np.isfinite(want)
    return (np.array_equal(np.isnan(got), np.isnan(want)) and np.array_equal(got[np.isinf(want)], want[np.isinf(want)])
            and np.all(np.abs(got[finite] - want[finite]) <= rel * (np.abs(want[finite]).max() if finite.any() else 1)))


def plant_specials(a, seed, also=(), largest=True):
    """A copy of `a` with an infinity of each sign, NaNs (quiet, of all ones, signalling with a low bit), a zero and the
    largest numbers at places that the seed picks (and at the flat places `also`).  Without `largest` where two operands have
    them: whether a sum of two products above the largest number overflows depends on the order."""
    a = np.ascontiguousarray(a, np.float32).copy()
    flat = a.reshape(-1).view(np.uint32)
    values = np.array([0x7F800000, 0xFF800000, 0x7FC00000, 0x7FFFFFFF, 0x7F800001, 0x00000000, 0x7F7FFFFF, 0xFF7FFFFF][:8 if largest else 6], np.uint32)
    at = np.random.default_rng(seed).choice(flat.size, size=min(len(values), flat.size), replace=False)
    flat[at] = values[:len(at)]
    for i, k in enumerate(also):
        flat[k] = values[i % 2]
    return a


def dev(a):
    import torch

    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()


def host(t):
    return t.detach().cpu().numpy()
