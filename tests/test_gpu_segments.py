"""Byte-filter scans that take long sequences in segments (bit-exact against the oracle).

Few sequences, some of them very long, make a launch cut its long sequences
into segments that different lane groups score.  Planted hits near and
across segment ends, several hits in one sequence (J chaining: the rescoring
kernel visits some segments and skips others), overflows, and sequences just
around a segment's length, over kernels of every kind.
"""
import numpy as np
import pytest

from paper_1707_09683_gb300 import synth

pytestmark = pytest.mark.gpu


def long_database(profs, rng, lengths):
    lengths = np.asarray(lengths, dtype=np.uint32)
    offsets = np.concatenate([[0], np.cumsum(lengths[:-1], dtype=np.uint64)]).astype(np.uint64)
    db = synth.Database(residues=synth.draw_residues(int(lengths.sum()), rng), offsets=offsets, lengths=lengths)
    for s in range(lengths.size):          # weak and strong hits, anywhere, some sequences with many
        for _ in range(int(rng.integers(0, 8))):
            p = profs[int(rng.integers(len(profs)))]
            n = int(min(rng.integers(12, 40), p.M, lengths[s]))
            if n < 1:
                continue
            k, w = int(rng.integers(0, p.M - n + 1)), int(rng.integers(0, lengths[s] - n + 1))
            for j in range(n):
                e = p.emit[k + j]
                db.residues[int(offsets[s]) + w + j] = rng.choice(20, p=e / e.sum()) if rng.random() < 0.6 else int(e.argmax())
    return db


def compare(profs, db, config=None, f16=False):
    import torch

    import oracle
    from paper_1707_09683_gb300 import mpf

    ctx = mpf.Context(0)
    ps = [mpf.Profile(ctx, p) for p in profs]
    for p in ps:
        for f in (mpf.MSV, mpf.SSV):
            if config:
                p.set_config(f, *config)
            if f16:
                p.set_arith(f, mpf.ARITH_F16)
    ddb = mpf.Database(ctx, db.residues, db.offsets, db.lengths)
    n, q = db.n_seqs, len(ps)
    want = [[f(p, db.residues, db.offsets, db.lengths, nthreads=16) for p in profs] for f in (oracle.msv, oracle.ssv)]
    for filt in (mpf.MSV, mpf.SSV, mpf.MSV_SSV):
        blocks = want if filt == mpf.MSV_SSV else [want[filt]]
        out = [torch.full((len(blocks) * q * n,), 99, dtype=t, device="cuda")
               for t in (torch.uint8, torch.uint8, torch.float32)]
        plan = mpf.Plan(ctx, filt, ps, ddb, *out)
        for graph in (False, True):        # twice: the counters start from zero each time
            if graph:
                plan.capture_graph()
            for t in out:
                t.fill_(99)
            torch.cuda.synchronize()
            plan.launch()
            ctx.sync()
            for j in range(3):
                exp = np.concatenate([w[j] for b in blocks for w in b])
                np.testing.assert_array_equal(out[j].cpu().numpy(), exp, err_msg=f"filter {filt} output {j}")
    return want


@pytest.mark.parametrize("M,config", [(30, None), (100, None), (100, (32, 4)), (400, None), (777, None),
                                      (777, (32, 14)), (777, (32, 26)), (1500, None), (3000, None)])
def test_long_sequences_in_segments(M, config):
    rng = np.random.default_rng(M + (config[1] if config else 0))
    profs = [synth.make_profile(M, rng)]
    S = max(128, (M + 3) // 4 * 4)
    lengths = [S - 1, S, S + 1, S + 3, 2 * S - 1, 2 * S, 2 * S + 1, 5 * S + 2, 9 * S, 20000, 7001, 35000, 0, 1, 300]
    want = compare(profs, long_database(profs, rng, lengths), config)
    flags = np.concatenate([w[1] for w in want[0]])
    assert (flags == 0).any()


def test_segments_in_batches_and_with_fp16_cells():
    rng = np.random.default_rng(5)
    profs = [synth.make_profile(M, rng) for M in (150, 140, 160, 155, 60, 900, 2100)]
    db = long_database(profs, rng, [30000, 12000, 5000, 700, 650, 640, 500, 10, 9000])
    compare(profs, db)
    compare(profs[5:6], db, f16=True)
