"""Exact MSV rescoring of many listed sequences, several to a warp (bit-exact
against the oracle).

With more listed sequences than the launch on 32 lanes takes, narrow groups
of a warp rescore different sequences in lock step.  Sequences cut into
segments, with hits in neighbouring segments and across their ends, stand
beside sequences whose first hit lies later and beside short ones, so the
groups' segments end at different rows.
"""
import numpy as np
import pytest

from paper_1707_09683_gb300 import synth

pytestmark = pytest.mark.gpu

M, N_SHORT, N_LONG = 90, 10000, 1200


@pytest.fixture(scope="module")
def workload():
    import oracle

    rng = np.random.default_rng(17)
    recs = [synth.make_profile(M, rng) for _ in range(2)]
    lengths = np.concatenate([np.full(N_SHORT, 100), rng.integers(1500, 9000, N_LONG)]).astype(np.uint32)
    offsets = np.concatenate([[0], np.cumsum(lengths[:-1], dtype=np.uint64)]).astype(np.uint64)
    res = synth.draw_residues(int(lengths.sum()), rng)
    best = [r.emit.argmax(axis=1).astype(np.uint8) for r in recs]

    def hit(s, at, which, n):
        k = int(rng.integers(0, M - n + 1))
        seg = best[which][k:k + n].copy()
        noise = rng.random(n) < 0.35
        seg[noise] = synth.draw_residues(int(noise.sum()), rng)
        res[int(offsets[s]) + at:int(offsets[s]) + at + n] = seg

    for s in range(lengths.size):
        for which in range(2):
            if s < N_SHORT:
                hit(s, 50 * which + int(rng.integers(0, 26)), which, 28)
            else:
                for _ in range(int(rng.integers(1, 6))):
                    n = int(rng.integers(20, 36))
                    hit(s, int(rng.integers(0, lengths[s] - n)), which, n)
    db = synth.Database(residues=res, offsets=offsets, lengths=lengths)
    want = [[f(r, res, offsets, lengths, nthreads=16) for r in recs] for f in (oracle.msv, oracle.ssv)]
    # Sequences that the held pass lists: largest cell above T, below overflow.
    for r, (raw, _, _) in zip(recs, want[1]):
        t = r.tjb_by_len[np.minimum(lengths, r.tjb_by_len.size - 1)].astype(int)
        b = r.base - t - r.tbm
        listed = (raw > r.base + r.tec - b) & (raw < 255 - r.bias - b)
        assert listed.sum() > 48 * 160 and listed[N_SHORT:].sum() > N_LONG // 3
    return recs, db, want


@pytest.mark.parametrize("lanes,words,queries,f16", [
    (1, 46, 1, False), (2, 24, 1, False), (4, 12, 1, False), (8, 6, 1, False), (16, 4, 1, False),
    (8, 6, 1, True), (16, 4, 1, True), (16, 8, 2, False), (0, 0, 1, False), (0, 0, 2, False)])
def test_many_listed_sequences(workload, lanes, words, queries, f16):
    import torch

    from paper_1707_09683_gb300 import mpf

    recs, dbh, want = workload
    ctx = mpf.Context(0)
    db = mpf.Database(ctx, dbh.residues, dbh.offsets, dbh.lengths)
    profs = [mpf.Profile(ctx, r) for r in recs[:queries]]
    for p in profs:
        for f in (mpf.MSV, mpf.SSV):
            if lanes:
                p.set_config(f, lanes, words)
            if f16:
                p.set_arith(f, mpf.ARITH_F16)
    n = db.n_seqs
    for filt in (mpf.MSV, mpf.MSV_SSV):
        blocks = want if filt == mpf.MSV_SSV else want[:1]
        out = [torch.full((len(blocks) * queries * n,), 99, dtype=t, device="cuda")
               for t in (torch.uint8, torch.uint8, torch.float32)]
        mpf.scan_batch(ctx, filt, profs, db, *out)
        ctx.sync()
        for j in range(3):
            exp = np.concatenate([w[j] for b in blocks for w in b[:queries]])
            got = out[j].cpu().numpy()
            assert np.array_equal(got, exp), (filt, j, np.flatnonzero(got != exp).size)
