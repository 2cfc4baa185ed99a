"""Near ties of the two-level race's first level, for tests of the drafters'
log-domain keys.

A row holds two blocks with weight: one entry of block a at the logit MA, and
all 256 entries of block b at MB.  The winner is the sign of
    log2 E_a - log2 E_b - (MA - MB) log2(e) / tau + 8,
evaluated here in 64 bits over many request ids; the ids returned are those
within `bound` of a tie and further than `margin` from it.

bound: what a key loses if its block sum is relative to the rounded product
fl(M c2) and its max is compared by the exact one, |rho_a - rho_b| with
rho = M c2 - fl(M c2).
margin: the errors a key may have.  log2 of E (|log2 E| <= 24) and of the sum
(of 256 equal terms) by lg2.approx, at most 2^-22 of the result each (2^-22
absolute next to 1): 24 * 2^-22 + 8 * 2^-22; log1p, ex2.approx, the sum's
roundings and the key's subtractions, each at most 2^-22 of values up to 32 in
all: 8 * 2^-22.  Two keys: 80 * 2^-22 < 2e-5.
"""
import numpy as np

MARGIN = 2e-5
TAU = np.float32(0.0095)
MA, MB = 13.9375, 13.875  # (MA - MB) log2(e) / TAU = 9.5
NONE = -1e4              # a logit without weight at TAU
SEED, POSITION = 77, 100
PURPOSE_DRAFT = 4


def philox(ctr, k0, k1):
    """Philox4x32-10 of four counter arrays (uint64 holding 32-bit words)."""
    low = np.uint64(0xFFFFFFFF)
    c = [np.asarray(x, np.uint64) for x in ctr]
    for _ in range(10):
        p0, p1 = np.uint64(0xD2511F53) * c[0], np.uint64(0xCD9E8D57) * c[2]
        c = [(p1 >> np.uint64(32)) ^ c[1] ^ np.uint64(k0), p1 & low,
             (p0 >> np.uint64(32)) ^ c[3] ^ np.uint64(k1), p0 & low]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return c


def block_variate(ids, block):
    """log2 E of a race block for each request id, at draft 0."""
    n = len(ids)
    ctr = [np.full(n, POSITION + 1), ids & np.uint64(0xFFFFFFFF), ids >> np.uint64(32),
           np.full(n, PURPOSE_DRAFT << 28 | block >> 2)]
    word = philox(ctr, SEED, 0)[block & 3]
    u = (2 * (word >> np.uint64(9)).astype(np.float64) + 1) * 2.0**-24
    return np.log2(-np.log(u))


def find(a, b, n=1 << 20):
    """(request ids, the winning block of each)."""
    c2 = 1.4426950408889634 / float(TAU)
    c2f = np.float32(c2)
    rho = [M * float(c2f) - float(np.float32(M) * c2f) for M in (MA, MB)]
    bound = abs(rho[0] - rho[1])
    ids = np.arange(1, n + 1, dtype=np.uint64)
    d = block_variate(ids, a) - block_variate(ids, b) - (MA - MB) * c2 + 8.0
    near = (np.abs(d) > MARGIN) & (np.abs(d) < bound - MARGIN)
    return ids[near], np.where(d[near] < 0, a, b)


def row(V, a, b):
    """The row's logits."""
    x = np.full(V, NONE, np.float32)
    x[256 * a + 17] = MA
    x[256 * b:256 * b + 256] = MB
    return x
