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
