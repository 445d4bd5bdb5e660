"""The pruned beam search against the search without pruning, bit for bit, on inputs whose scores are not exact in
fp32 (aq_beam_search, Alg. 1 and App. C): Gaussian weights, scores that cancel almost completely, channels of
very different energy, codebooks and scales far from 1.

The search without pruning is the same kernel where its magnitudes are beyond the estimates' range: H times a
power of two scales every fp32 term, sum and score exactly, so the codes stay the same, and from 1e36 < 2^120 on
every candidate is scored by the definition. A group is compared at a power that brings a lower bound of its
magnitudes T (the kernel's comment) above 2^120 and keeps an upper bound below 2^130: that bound adds the
largest entries of all books in every element, while a state has already used up the earlier books to
approach the weights, so the sums themselves stay below a sixteenth of it (and E_k S below 2^126)."""
import numpy as np
import pytest

import aq_testutil as U
import oracle
import workloads
from test_gpu_beam import run_beam

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def gpu():
    U.require_gpu()


def widen(bits, dt):
    b = np.asarray(bits, np.uint16)
    return (b.view(np.float16) if dt == "f16" else (b.astype(np.uint32) << 16).view(np.float32)).astype(np.float64)


def bounds(layer, W, H, lam):
    """Bounds of the terms of a group's scores over the books, [out][groups]: from below, from above, and of the
    sums E_k S."""
    out, inp, M, dt = layer["out"], layer["in"], layer["M"], layer["book_dtype"]
    S = (H + H.T) / 2
    books, s = np.abs(widen(layer["books"], dt)), np.abs(widen(layer["scales"], dt))
    cmax = books.max(axis=1)                                         # [M][8]
    low, up, score, cross = np.inf, 0.0, 0.0, 0.0
    prefix = np.zeros((out, inp))
    for k in range(M):
        prefix += widen(layer["books"], dt)[k][layer["codes"][:, :, k]].reshape(out, inp)
        E = W - widen(layer["scales"], dt)[:, None] * prefix
        V = E @ S
        cross = np.maximum(cross, (np.abs(E) @ np.abs(S)).reshape(out, inp // 8, 8).max(axis=2))
        lo, hi = np.zeros((out, inp // 8)), np.zeros((out, inp // 8))
        for g in range(inp // 8):
            Sg = S[g * 8:g * 8 + 8, g * 8:g * 8 + 8]
            h = np.abs(V[:, g * 8:g * 8 + 8] - E[:, g * 8:g * 8 + 8] @ Sg)
            w = np.abs(W[:, g * 8:g * 8 + 8])
            for D, t in ((w + s[:, None] * cmax[k], lo), (w + s[:, None] * cmax[:k + 1].sum(0), hi)):
                t[:, g] = np.einsum("oi,ij,oj->o", D, np.abs(Sg), D) + 2 * (D * h).sum(1)
        low = np.minimum(low, lam[k] * lo)
        score = score + lam[k] * hi
        up = np.maximum(up, lam[k] * hi + score)
    return low, up, cross


CASES = {
    # kind: (out, in, M, dtype, weight std, book std, scale, H channel spread in powers of 10, lambda)
    "gaussian": (96, 96, 4, "f16", 0.04, 0.02, 1.0, 0.0, [1.0, 0.5, 0.25, 0.125]),
    "cancelling": (96, 96, 3, "f16", 30.0, 0.002, 1.0, 0.0, [1.0, 1.0, 1.0]),
    "channels": (64, 128, 3, "bf16", 40.0, 20.0, 1.0, 1.0, [1.0, 2.0, 3.0]),
    "books far from 1": (64, 64, 3, "bf16", 0.04, 0.02 * 2.0 ** 68, 2.0 ** -68, 0.0, [1.0, 1.0, 1.0]),
    "books near 0": (64, 64, 3, "bf16", 0.04, 0.02 * 2.0 ** -60, 2.0 ** 60, 0.0, [1.0, 1.0, 1.0]),
}


@pytest.mark.parametrize("K", [1, 8, 16])
@pytest.mark.parametrize("kind", sorted(CASES))
def test_pruned_equals_full_search(kind, K):
    out, inp, M, dt, wstd, bstd, scale, spread, lam = CASES[kind]
    rng = np.random.Generator(np.random.PCG64(len(kind)))
    layer = dict(out=out, **{"in": inp}, G=8, M=M, B=8, book_dtype=dt, scale_dtype=dt,
                 books=workloads.to_bits((rng.standard_normal((M, 256, 8)) * bstd).astype(np.float32), dt),
                 codes=rng.integers(0, 256, size=(out, inp // 8, M), dtype=np.uint8),
                 scales=workloads.to_bits((rng.uniform(0.5, 1.5, out) * scale).astype(np.float32), dt))
    W_bits = workloads.to_bits((rng.standard_normal((out, inp)) * wstd).astype(np.float32), dt)
    X = rng.standard_normal((inp, 3 * inp)) * 10.0 ** rng.uniform(-spread, spread, (inp, 1))
    H = ((X @ X.T) / (3 * inp)).astype(np.float32).astype(np.float64)
    got = run_beam(layer, W_bits, H, lam, K)
    low, up, cross = bounds(layer, widen(W_bits, dt), H, lam)
    seen = np.zeros(low.shape, bool)
    for e in range(30, 200, 2):
        here = (up * 2.0 ** e < 2.0 ** 130) & (low * 2.0 ** e > 2.0 ** 120) & (cross * 2.0 ** e < 2.0 ** 126) & ~seen
        if not here.any() or np.abs(H).max() * 2.0 ** e >= 2.0 ** 127:
            continue
        full = run_beam(layer, W_bits, H * 2.0 ** e, lam, K)
        assert np.array_equal(got[here], full[here]), "%d of %d groups differ at 2^%d" % (
            int((got[here] != full[here]).any(axis=-1).sum()), int(here.sum()), e)
        seen |= here
    assert seen.mean() >= 0.5, "only %.2f of the groups could be compared" % seen.mean()
