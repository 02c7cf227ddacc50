"""Byte filters on long weak diagonals (bit-exact against the oracle).

The striped integer kernels take rows in pairs: the first row's sums are
32-bit additions of packed cells, whose carries collect in the fraction bits
of the upper cell and are cleared every 120 rows.  Scores of -1, 0 and 1
keep diagonals alive for hundreds of rows, a carry in most of them, so a
carry that reached a score unit would change the result.  Databases without
code 20 or above (at most 21 table rows in tensor memory) and with them take
different kernels.
"""
import numpy as np
import pytest

from paper_1707_09683_gb300 import synth

pytestmark = pytest.mark.gpu

# (lanes, words): shared-memory tables at every lane count, tensor-memory
# tables held whole (up to 14 or 24 words) and split with shared memory.
CONFIGS = [(1, 48), (2, 48), (4, 40), (8, 26), (16, 18), (32, 4), (32, 8), (32, 10), (32, 14), (32, 16),
           (32, 18), (32, 22), (32, 24), (32, 26), (32, 30), (32, 38), (32, 48)]


def weak_profile(M, rng, K):
    p = synth.random_profile(M, K, rng, bias=3, tbm=40, tec=3, tjb=20, base=190)
    p.cost[:] = rng.choice([2, 3, 4], size=p.cost.shape, p=[0.32, 0.33, 0.35]).astype(np.uint8)
    return p


@pytest.mark.parametrize("codes", [20, 21, 32])
@pytest.mark.parametrize("lanes,words", CONFIGS)
def test_long_weak_diagonals(lanes, words, codes):
    rng = np.random.default_rng(1000 * lanes + words + codes)
    check(2 * lanes * words - (words > 4) * int(rng.integers(0, 2 * lanes)), codes, rng, lanes, words)


@pytest.mark.parametrize("M", [3073, 4100, 5000])
def test_long_weak_diagonals_across_tiles(M):
    """Models past the striped table: diagonals cross from tile to tile."""
    check(M, 20, np.random.default_rng(M))


@pytest.mark.parametrize("codes", [20, 25, 26])
@pytest.mark.parametrize("M", [3073, 3840, 4096, 4100])
def test_tile_rows_left_over_after_turns_of_eight(M, codes):
    """Every remainder of a tile's turns of eight rows, before and around a
    clearing row; tiles of 16 and 20 words (the latter hold 25 codes)."""
    check(M, codes, np.random.default_rng(8 * M), lengths=[*range(20), *range(112, 130), 1201])


LENGTHS = [3, 119, 120, 121, 122, 240, 243, 1201, 0, 1, 777, 2, 1802]


def check(M, codes, rng, lanes=0, words=0, lengths=LENGTHS):
    import torch

    import oracle
    from paper_1707_09683_gb300 import mpf

    p = weak_profile(M, rng, codes)
    lengths = np.array(lengths, dtype=np.uint32)
    offsets = np.concatenate([[0], np.cumsum(lengths[:-1])]).astype(np.uint64)
    res = rng.integers(0, codes, size=int(lengths.sum())).astype(np.uint8)
    res[0] = codes - 1
    n = lengths.size
    ctx = mpf.Context(0)
    prof, db = mpf.Profile(ctx, p), mpf.Database(ctx, res, offsets, lengths)
    for filt in (mpf.MSV, mpf.SSV):
        if words:
            prof.set_config(filt, lanes, words)
    want = [f(p, res, offsets, lengths) for f in (oracle.msv, oracle.ssv)]
    for filt, fn in ((mpf.MSV, mpf.msv_scan), (mpf.SSV, mpf.ssv_scan)):
        out = [torch.full((n,), 99, dtype=t, device="cuda") for t in (torch.uint8, torch.uint8, torch.float32)]
        fn(ctx, prof, db, *out)
        ctx.sync()
        for got, exp in zip(out, want[filt]):
            np.testing.assert_array_equal(got.cpu().numpy(), exp)
    both = [np.zeros(2 * n, dtype=t) for t in (np.uint8, np.uint8, np.float32)]
    mpf.scan_batch(ctx, mpf.MSV_SSV, [prof], db, *both)
    for j in range(3):
        np.testing.assert_array_equal(both[j], np.concatenate([want[0][j], want[1][j]]))
