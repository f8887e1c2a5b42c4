"""The rule behind the threshold x-step's list, checked on the host against the FP64 oracle.

The x-step lists the entries of v above a lower bound G of the operator's threshold and works on the list.
G comes from last sweep's threshold or from the maxima of 512 (j up to 170) or 2048 subsets of v
(kernel_xstep.cu).  The model here makes the subsets as the threads of a CTA of 128, 256, 512 or 1024 do, from
rows at every alignment, bins their maxima, takes the edge of the bin of the j-th largest, lists by 16 segments of at most 64 entries, and accepts the list as the kernel
does (at least s or s + 1 entries; phi(G) < 0 for lambda_s, where a sample of phi over the maxima picks j).
The bound has to be the same for every CTA size and alignment, and the x-step on an accepted list, scattered back, the
x-step on all of v."""
import numpy as np
import pytest

BINS, SHIFT, COARSE_J, COARSE_MAX_J, MAX_J, CAND, SEG_CAP = 2048, 17, 170, 200, 500, 1024, 64
COARSE, FINE = 512, 2048


def keys(a):
    return np.abs(a).astype(np.float32).view(np.uint32).astype(np.int64)


def value(key):
    return float(np.uint32(key).view(np.float32))


def subset_maxima(k, T, N, shift=0):
    """Maxima of N subsets as a CTA of T threads forms them from a row that begins `shift` entries into a vector:
    thread t loads the four entries from 4 t + 4 T h on, h = 0, 1, ...; load h goes to its group h mod G of four
    subsets, and group g's e-th is subset (4 (t + T g) + e) mod N."""
    G = max(1, N // (4 * T))
    m = np.zeros(N, np.int64)
    q = np.arange(k.size) + shift
    h, rest = np.divmod(q, 4 * T)
    t, e = np.divmod(rest, 4)
    np.maximum.at(m, (4 * (t + T * (h % G)) + e) % N, k)
    return np.sort(m)


def histogram(maxima):
    top = int(maxima.max())
    return np.bincount(np.minimum((top - maxima) >> SHIFT, BINS - 1), minlength=BINS), top


def rank_bin(hist, j):
    return min(int(np.searchsorted(np.cumsum(hist), j)), BINS - 1)


def edge(top, b):
    down = (b + 1) << SHIFT
    return 0 if b >= BINS - 1 or down >= top else top - down


def root_above(hist, top, b, s, p, N):
    G = edge(top, b)
    if G == 0:
        return True
    w = np.array([value(top - (q << SHIFT) - (1 << (SHIFT - 1))) - value(G) for q in range(b + 1)])
    n, w1, w2 = hist[:b + 1].sum(), (hist[:b + 1] * w).sum(), (hist[:b + 1] * w * w).sum()
    q = max(1.0, p / N)
    m = N * q * (1.0 - (1.0 - n / N) ** (1.0 / q))
    return s * w2 < 1.02 * (m / n) * w1 * w1


def bound(hists, j, lam_s, p):
    """(G's key, j) or None; hists: (histogram, largest maximum) of 512 and of 2048 subsets."""
    for N, limit, (hist, top) in zip((COARSE, FINE), (COARSE_MAX_J, MAX_J), hists):
        if N == COARSE and j > COARSE_J:
            continue
        b = rank_bin(hist, j)
        while lam_s > 0 and b is not None and not root_above(hist, top, b, lam_s, p, N):
            longer = j < limit
            j = min(limit, j + j // 2)
            b = rank_bin(hist, j) if longer else None
        if b is not None:
            return edge(top, b), j
    return None


def list_above(k, G):
    """Indices of the entries above G, or None when a segment holds too many."""
    at = np.flatnonzero(k > G)
    if k.size > CAND:
        seg = ((k.size + 15) // 16 + 127) // 128 * 128
        if np.bincount(at // seg, minlength=16).max() > SEG_CAP:
            return None
    return at


def phi(a, s, G):
    w = a[a > G] - G
    return s * np.sum(w * w) - np.sum(w) ** 2


def vectors(rng, p):
    yield rng.standard_normal(p)
    yield rng.standard_t(2, p)                                                  # heavy tails
    v = rng.standard_normal(p); v[::5] = 0.0; yield v                           # exact zeros
    v = rng.standard_normal(p); v[p // 3:p // 3 + p // 20] = v[7]; yield v      # a run of equal magnitudes
    v = rng.standard_normal(p) * 0.05; v[rng.choice(p, p // 80, replace=False)] += 3; yield v
    v = rng.standard_normal(p); v[p // 2:p // 2 + p // 16] *= 20; yield v       # crowded into one segment


@pytest.mark.parametrize("p", [70, 1000, 1027, 3001, 9000])
@pytest.mark.parametrize("form", range(1, 9))
def test_list_gives_the_full_x_step(oracle, form, p):
    rng = np.random.default_rng(31 * form + p)
    accepted = left = 0
    for v in vectors(rng, p):
        v = v.astype(np.float32).astype(np.float64)
        k, a = keys(v), np.abs(v)
        hists = []
        for N in (COARSE, FINE):                              # the bound depends on neither CTA size nor alignment
            bases = [subset_maxima(k, T, N, shift) for T in (128, 256, 512, 1024) for shift in range(4)]
            assert all(np.array_equal(bases[0], other) for other in bases[1:])
            hists.append(histogram(bases[0]))
        for s in (1, 12, 60, 150, 400):
            if form not in (3, 4) and (s + (form > 4)) * 6 > p:
                continue
            if s > p:
                continue
            calibrate = form >= 5
            need = s + 1 if calibrate else s
            full = oracle.xstep(form, v, float(s), 0.0, calibrate)
            thr = abs(full.thr) if form in (3, 4) else float(np.sort(a)[::-1][need - 1])
            lam = s if form in (3, 4) else 0
            got = bound(hists, min(3 * s + 16, MAX_J) if lam else need, lam, p)
            tries = [] if got is None else [got[0]]
            tries += [int(keys(np.array([f * thr]))[0]) for f in (0.6, 0.85, 0.95, 1.0, 1.1)]   # last sweep's
            for G in tries:
                at = list_above(k, G)
                g = value(G)
                if at is None or (lam and not (phi(a[at], s, g) < 0)) or (not lam and at.size < need and G > 0):
                    left += 1
                    continue
                accepted += 1
                part = oracle.xstep(form, v[at], float(min(s, at.size)) if form <= 2 else float(s), 0.0,
                                    calibrate and at.size >= need) if at.size else None
                if part is None:
                    continue
                x = np.zeros(p)
                x[at] = part.x
                if not lam and at.size < need:
                    continue                                  # fewer nonzero entries than are selected: all of them
                assert np.array_equal(x, full.x), (s, G)
                assert part.F == full.F and part.nnz == full.nnz and part.thr == full.thr
    assert accepted > 0 and left > 0


def test_bound_lists_at_least_j_and_not_many_more():
    rng = np.random.default_rng(8)
    over = 0
    for _ in range(30):
        k = keys(rng.standard_normal(20000))
        hists = [histogram(subset_maxima(k, 512, N)) for N in (COARSE, FINE)]
        for j in (10, 100, COARSE_J, COARSE_J + 1, 300, MAX_J):
            G, _ = bound(hists, j, 0, k.size)
            n = int((k > G).sum())
            assert j <= n < 1.4 * j + 20                      # a bin is 2^-6 octave wide
            over += list_above(k, G) is None
    assert over <= 2                                          # a segment rarely holds more than it may list
