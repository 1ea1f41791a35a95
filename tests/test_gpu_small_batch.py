"""Small ASCII batches packed and filtered by one launch, and the plain
launch's tiles per CTA, against the oracle."""
import numpy as np
import pytest

import oracle
from gpu_util import assert_same, to_dev, torch_cuda
from paper_1910_09020_gb300 import binding, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def F():
    torch_cuda()
    f = binding.Filter(0)
    yield f
    f.close()


@pytest.mark.parametrize("shift", [0, 1, 5])
@pytest.mark.parametrize("m", [1, 15, 16, 17, 33, 100, 128, 129, 255, 256])
def test_ascii_batch_matches_oracle(F, m, shift):
    """Every pair at sizes around a CTA's tile, every kind of route, ASCII
    that starts at any byte (shift), one launch per batch."""
    torch = torch_cuda()
    for n in (1, 127, 128, 129, 1000):
        reads, refs = synth.pairs_fixed(70 + m, 0, n, m,
                                        synth.rate_recipe(0.12))
        sides = []
        for side in (reads, refs):
            buf = torch.zeros(n * m + shift, dtype=torch.uint8, device="cuda")
            buf[shift:] = to_dev(side.reshape(-1))
            sides.append(buf[shift:])
        for E in (0, 1, 4, 5, 6, 15, 16, 31):
            before = F.counters().launches
            acc, obs = F.filter(*sides, m=m, e=E, n=n,
                                fmt=binding.SS_FMT_ASCII, sync=True)
            assert F.counters().launches == before + 1
            oacc, oobs = oracle.filter_batch(reads, refs, m, E)
            assert_same(acc.cpu().numpy(), obs.cpu().numpy(), oacc, oobs,
                        f"m={m} n={n} E={E} shift={shift}")


def test_ascii_batch_latches_a_bad_base(F):
    reads, refs = synth.pairs_fixed(71, 0, 300, 100, synth.SHORT_UNIFORM_K)
    for p, side in ((0, 0), (299, 1)):
        bad = [reads.copy(), refs.copy()]
        bad[side][p, 99] = ord("N")
        F.filter(to_dev(bad[0].reshape(-1)), to_dev(bad[1].reshape(-1)),
                 m=100, e=5, n=300, fmt=binding.SS_FMT_ASCII)
        with pytest.raises(binding.SSError) as ei:
            F.sync()
        assert ei.value.code == binding.SS_ERR_INVALID_BASE


@pytest.mark.parametrize("n", [299_999, 300_000, 300_001])
def test_ascii_batch_either_side_of_the_rule(F, n):
    """The last batch of one launch and the first of three: the same results,
    and those of the packed form."""
    torch = torch_cuda()
    m = 100
    reads, refs = synth.pairs_fixed(72, 0, n, m, synth.rate_recipe(0.12))
    q, r = to_dev(reads.reshape(-1)), to_dev(refs.reshape(-1))
    pq, pr = F.pack(q, m=m, n=n), F.pack(r, m=m, n=n)
    for E in (0, 5, 12):
        got = F.filter(q, r, m=m, e=E, n=n, fmt=binding.SS_FMT_ASCII)
        want = F.filter(pq, pr, m=m, e=E, n=n)
        F.sync()
        assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])


@pytest.mark.parametrize("tiles", [1, 799, 1601, 6401, 12799, 12801, 51201])
def test_tiles_per_cta(F, tiles):
    """Batches either side of the steps in a CTA's number of tiles, each with
    a last tile that is not full: the packed plain launch equals the
    bit-sliced one."""
    torch = torch_cuda()
    m, n = 64, tiles * 128 - 3
    g = torch.Generator(device="cuda")
    g.manual_seed(tiles)
    letters = torch.tensor([65, 67, 71, 84], dtype=torch.uint8, device="cuda")
    q = letters[torch.randint(0, 4, (n * m,), device="cuda", generator=g)]
    edit = torch.rand(n * m, device="cuda", generator=g) < 0.05
    r = torch.where(edit, letters[torch.randint(0, 4, (n * m,), device="cuda",
                                                generator=g)], q)
    pq, pr = F.pack(q, m=m, n=n), F.pack(r, m=m, n=n)
    sq, sr = F.pack_sliced(q, m=m, n=n), F.pack_sliced(r, m=m, n=n)
    for E in (0, 1, 3, 6):
        got = F.filter(pq, pr, m=m, e=E, n=n)
        want = F.filter(sq, sr, m=m, e=E, n=n, fmt=binding.SS_FMT_SLICED2)
        F.sync()
        assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
