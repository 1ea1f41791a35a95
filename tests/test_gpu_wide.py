"""GPU parity of the routes above 31 edits with the oracle: every class at
its bounds, few and many pairs of a class, repeats (which the index and the
ring teams hand over to all rows) and accurate pairs."""
import numpy as np
import pytest

import oracle
from gpu_util import assert_same, to_dev, torch_cuda
from paper_1910_09020_gb300 import binding, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def F():
    torch_cuda()
    f = binding.Filter(0, workspace_bytes=2 << 30)
    yield f
    f.close()


def noisy(rng, seq, rate):
    """seq (codes) with substitutions, insertions and deletions, of its
    length."""
    n = len(seq)
    u = rng.random(n)
    out = np.where(u < rate / 3, rng.integers(0, 4, n), seq)
    times = np.where(u < rate / 3, 1,
                     np.where(u < 2 * rate / 3, 2, np.where(u < rate, 0, 1)))
    out = np.repeat(out, times)
    extra = rng.integers(0, 4, max(0, n - len(out)))
    return np.concatenate([out, extra])[:n]


def pair(rng, kind, m, rate):
    """A pair of m bases: kind 0 random, 1 to 3 a repeat of 1, 2 or 171 bases
    with errors on either side, 4 a repeat between random bases."""
    if kind in (0, 4):
        base = rng.integers(0, 4, m)
        if kind == 4:
            a, b = m // 3, m // 3 + m // 4
            base[a:b] = np.resize([0, 1], b - a)
        return base, noisy(rng, base, rate)
    base = np.resize(rng.integers(0, 4, (0, 1, 2, 171)[kind]), m)
    return noisy(rng, base, 0.05), noisy(rng, base, rate)


def batch(F, cases, seed):
    """cases: (kind, m, rate, E) each.  Routes them on the GPU; returns its
    and the oracle's results."""
    torch = torch_cuda()
    rng = np.random.default_rng(seed)
    sides = [pair(rng, k, m, rate) for k, m, rate, _ in cases]
    L = np.array([c[1] for c in cases], np.int32)
    Es = np.array([c[3] for c in cases], np.int32)
    off = np.concatenate([[0], np.cumsum(L, dtype=np.int64)])
    words = (L.astype(np.int64) + 15) // 16
    woff = np.concatenate([[0], np.cumsum(words)])
    letters = np.frombuffer(b"ACGT", np.uint8)
    host, dev = [], []
    dL, doff, dwoff = to_dev(L), to_dev(off[:-1].copy()), to_dev(
        woff[:-1].copy())
    for k in (0, 1):
        a = letters[np.concatenate([s[k] for s in sides])]
        out = torch.zeros(int(woff[-1]), dtype=torch.int32, device="cuda")
        F.pack(to_dev(a), offsets=doff, lengths=dL, out=out,
               out_offsets=dwoff)
        host.append(a)
        dev.append(out)
    return host, off, L, Es, dev, dwoff, dL


def check(F, cases, seed, what, flags=0):
    host, off, L, Es, dev, dwoff, dL = batch(F, cases, seed)
    acc, obs = F.filter(dev[0], dev[1], offsets=dwoff, lengths=dL,
                        E=to_dev(Es), flags=flags, sync=True)
    oacc, oobs = oracle.filter_batch(host[0], host[1], L, Es, offsets=off)
    assert_same(acc.cpu().numpy(), obs.cpu().numpy(), oacc, oobs, what)
    return oacc


BOUNDS = [32, 112, 113, 304, 305, 511, 512, 816, 817, 1664, 1665, 5920, 5921,
          10016, 10017]


@pytest.mark.parametrize("flags", [0, binding.SS_FLAG_NO_GRAPH])
def test_class_bounds(F, flags):
    """Thresholds either side of every class bound, lengths around the words
    and rings and far above the threshold, accurate and rejected pairs, and
    thresholds above the length."""
    cases = []
    for e in BOUNDS:
        for m in sorted({e + 1, e + 2, e + 33, 2 * e + 5, 16384, 16385}):
            if m <= e:
                continue
            for rate in (0.01, 0.25):
                cases.append((0, m, rate, e))
    for m in (33, 113, 305, 817, 1665, 5921, 10017, 10018):
        cases.append((0, m, 0.3, m + 7))       # clamped to m - 1
    cases += [(0, 65536, 0.02, 3000), (0, 65537, 0.06, 7000),
              (0, 131072, 0.05, 10016), (0, 131072, 0.12, 10017),
              (0, 131072, 0.003, 500), (0, 131072, 0.01, 2000),
              (0, 131072, 0.1, 131071)]
    acc = check(F, cases, 3, "class bounds", flags)
    assert 0 < acc.mean() < 1


@pytest.mark.parametrize("kind", [1, 2, 3, 4])
def test_repeats(F, kind):
    """Repeats through every class above 31 edits: the index leaves them to
    all rows and, after the repeat of kind 4, goes on."""
    cases = [(kind, m, rate, e)
             for e in (40, 112, 300, 500, 816, 900, 1664, 3000, 8000, 12000)
             for m in (e + 40, 3 * e, 12 * e) if m < 60000
             for rate in (0.0, 0.02, 0.2)]
    check(F, cases, 10 + kind, f"repeats, kind {kind}")


def test_accurate_and_changing_pairs(F):
    """Long pairs whose steps are long (all rows) or short (the index), and
    pairs whose error rate changes on the way."""
    cases = [(0, m, rate, m * pm // 1000) for m in (30000, 100000)
             for rate in (0.0, 0.001, 0.01, 0.03, 0.15)
             for pm in (10, 20, 50, 100)]
    check(F, cases, 20, "accurate pairs")
    torch = torch_cuda()
    rng = np.random.default_rng(21)
    letters = np.frombuffer(b"ACGT", np.uint8)
    for e in (1500, 4000, 9000):
        q = rng.integers(0, 4, 10 * e)
        parts = [noisy(rng, x, rate) for x, rate in
                 zip(np.array_split(q, 6), (.005, .12, .01, .1, .002, .15))]
        r = np.concatenate(parts)
        qa, ra = letters[q], letters[r]
        m = len(q)
        dq, dr = (F.pack(to_dev(x), m=m, n=1) for x in (qa, ra))
        acc, obs = F.filter(dq, dr, m=m, e=e, n=1, sync=True)
        want = oracle.filter_pair(qa.tobytes(), ra.tobytes(), e)
        assert int(obs[0]) == want.obstacles
        assert bool(acc[0]) == want.accept
    torch.cuda.synchronize()


@pytest.mark.parametrize("m,e", [(400, 40), (700, 112), (900, 200),
                                 (1200, 310), (1500, 600)])
@pytest.mark.parametrize("n", [60, 3000, 30000])
def test_few_and_many_pairs(F, m, e, n):
    """One length and threshold: a pair to a warp, a pair to a team of lanes
    (30,000 pairs), among them repeats that a team hands over to its warp."""
    rng = np.random.default_rng(m + n)
    kinds = 60
    some = [pair(rng, (0, 0, 0, 1, 2, 3, 4)[k % 7], m,
                 (0.0, 0.01, 0.05, 0.15, 0.4)[k % 5]) for k in range(kinds)]
    letters = np.frombuffer(b"ACGT", np.uint8)
    reads = letters[np.stack([s[0] for s in some])]
    refs = letters[np.stack([s[1] for s in some])]
    oacc, oobs = oracle.filter_batch(reads, refs, m, e)
    pick = rng.integers(0, kinds, n)
    q = F.pack(to_dev(reads[pick].reshape(-1)), m=m, n=n)
    r = F.pack(to_dev(refs[pick].reshape(-1)), m=m, n=n)
    acc, obs = F.filter(q, r, m=m, e=e, n=n, sync=True)
    assert_same(acc.cpu().numpy(), obs.cpu().numpy(), oacc[pick], oobs[pick],
                f"n={n} m={m} e={e}")


@pytest.mark.parametrize("k", [4, 8, 16])
def test_subgrids_of_the_largest_thresholds(F, k):
    """Every subgrid of the CTA kernel, which only pairs above 10016 edits
    reach, in every length bound of its classes."""
    F.set_tuning(31, k)
    try:
        check(F, [(kind, m, rate, e) for kind in (0, 2)
                  for m, e in ((10050, 10020), (16384, 12000), (16385, 16384),
                               (40000, 11000), (65537, 10017))
                  for rate in (0.02, 0.3)], 40, f"subgrid {k}")
    finally:
        F.set_tuning(31, 8)


def test_served_pairs_above_the_index(F):
    """Requests with pairs above 10016 edits, up to the longest, among a
    stream of ordinary queued pairs: all of them go to the queue, and the
    results are the oracle's."""
    rng = np.random.default_rng(60)
    letters = np.frombuffer(b"ACGT", np.uint8)
    reqs = []
    for k in range(8):
        cases = [(0, m, 0.05, m // 10)
                 for m in rng.integers(6000, 30000, 12)]
        cases += [(0, int(m), 0.1, 60) for m in rng.integers(200, 4000, 12)]
        if k % 2 == 0:
            cases += [(0, 50000, 0.1, 12000), (2, 30000, 0.02, 11000),
                      (0, 20000, 0.4, 19999)]
        if k == 2:
            cases += [(0, 131072, 0.12, 10017), (0, 70000, 0.02, 30000)]
        sides = [pair(rng, c, int(m), rate) for c, m, rate, _ in cases]
        L = np.array([c[1] for c in cases], np.int32)
        E = np.array([c[3] for c in cases], np.int32)
        off = np.concatenate([[0], np.cumsum(L, dtype=np.int64)])
        reqs.append([letters[np.concatenate([s[i] for s in sides])]
                     for i in (0, 1)] + [L, E, off])
    queued = sum(int((np.minimum(r[3], r[2] - 1) > 511).sum()) for r in reqs)
    with binding.Server(0, hbm_budget_bytes=4 << 30, slots=2) as S:
        tickets = [S.submit(*r[:4]) for r in reqs]
        outs = []
        for t in tickets:
            assert S.wait(t, timeout_s=60.0) == binding.SS_OK
            outs.append(S.fetch(t))
        stats = S.stats()
    assert stats["long_pairs_queued"] == queued
    for (rc, a, o, _), r in zip(outs, reqs):
        assert rc == binding.SS_OK
        oa, oo = oracle.filter_batch(r[0], r[1], r[2], r[3], offsets=r[4])
        assert_same(a, o, oa, oo, "served")


def test_autotune_leaves_subgrids_that_nothing_reaches(F):
    """Without pairs above 10016 edits the subgrids do nothing: they are not
    timed (a third of the passes) and the default stays."""
    def passes(cases):
        host, off, L, Es, dev, dwoff, dL = batch(F, cases, 70)
        before = F.counters().launches
        _, k, _ = F.autotune(dev[0], dev[1], offsets=dwoff, lengths=dL,
                             E=to_dev(Es), reps=1)
        return F.counters().launches - before, k
    try:
        few, k = passes([(0, 3000, 0.1, 300), (0, 500, 0.1, 20)] * 20)
        all_, _ = passes([(0, 3000, 0.1, 300), (0, 12000, 0.1, 11000)])
        assert k == 8 and all_ == 3 * few > 0
    finally:
        F.set_tuning(31, 8)
