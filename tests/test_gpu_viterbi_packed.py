"""Packed P7Viterbi kernel (two nodes per register) against the oracle, bit-exact.

Model lengths around the layout's edges (64 nodes per word of a warp, up to
eight words per lane, teams of up to sixteen warps), and what the packed
words make special: sequences long enough that the entry score sinks to the
floor (the offset is lowered, more than once, down to the true -32768),
overflows early and after that, residue codes without match scores (at the
start, alone, in runs), match scores below the reach of one step, profiles
whose insert moves forbid lowering the offset, and profiles that do not
qualify (entry moves that differ, moves below the reach).
"""
import numpy as np
import pytest

from paper_1707_09683_gb300 import synth

pytestmark = pytest.mark.gpu

MODELS = [1, 2, 3, 33, 63, 64, 65, 129, 200, 321, 448, 449, 512, 513, 577, 1000, 1025, 1600, 2405, 3072, 3073, 5000, 8192]


def emitted(vp, rng, start, length):
    """Residues that the profile's match states start.. favour."""
    return np.array([int(np.argmax(vp.msc[:, k])) for k in range(start, min(vp.M, start + length))], dtype=np.uint8)


def database(vp, rng, longest):
    bg = synth.draw_residues
    seqs = [bg(int(n), rng) for n in rng.integers(1, 500, size=24)]
    seqs += [bg(longest, rng), bg(longest // 2 + 1, rng), bg(0, rng), bg(1, rng)]
    hit = emitted(vp, rng, 0, 300)
    for before in (0, 40, 1900, longest // 2):      # hits early, and after the offset was lowered
        seqs.append(np.concatenate([bg(before, rng), hit, bg(30, rng)]))
        seqs.append(np.concatenate([bg(before, rng), hit[:9], bg(200, rng)]))
    for n, codes in ((1, [25]), (60, [20, 25, 31]), (300, range(18, 23))):   # codes without match scores
        seqs.append(rng.choice(list(codes), size=n).astype(np.uint8))
    mixed = bg(400, rng)
    mixed[rng.random(400) < 0.1] = 25
    seqs += [mixed, np.concatenate([np.full(5, 30, np.uint8), bg(100, rng)])]
    lengths = np.array([s.size for s in seqs], dtype=np.uint32)
    offsets = np.concatenate([[0], np.cumsum(lengths[:-1], dtype=np.uint64)]).astype(np.uint64)
    return synth.Database(residues=np.concatenate(seqs), offsets=offsets, lengths=lengths)


def check(vps, db):
    import torch

    import oracle
    from paper_1707_09683_gb300 import mpf

    ctx = mpf.Context(0)
    n, nq = db.n_seqs, len(vps)
    out = [torch.full((nq * n,), 77, dtype=t, device="cuda") for t in (torch.int16, torch.uint8, torch.float32)]
    mpf.viterbi_scan(ctx, [mpf.VitProfile(ctx, v) for v in vps],
                     mpf.Database(ctx, db.residues, db.offsets, db.lengths), *out)
    ctx.sync()
    for q, v in enumerate(vps):
        want = oracle.viterbi(v, db.residues, db.offsets, db.lengths, nthreads=16)
        for got, exp in zip(out, want):
            np.testing.assert_array_equal(got[q * n:(q + 1) * n].cpu().numpy(), exp, err_msg=f"M={v.M}")
    return want


@pytest.mark.parametrize("M", MODELS)
def test_packed_scores(M):
    rng = np.random.default_rng(M)
    vp = synth.make_vit_profile(M, rng)
    db = database(vp, rng, 9000 if M <= 2405 else 5200)
    _, flag, _ = check([vp], db)
    if M >= 300:
        assert flag.any() and not flag.all()


@pytest.mark.parametrize("kind", ["impossible", "sticky_inserts", "loops", "entry", "far_moves", "low_base", "flat"])
def test_profiles_at_the_edge_of_the_packed_form(kind):
    rng = np.random.default_rng(len(kind))
    vps = [synth.make_vit_profile(M, rng) for M in (70, 530, 1400)]
    for vp in vps:
        if kind == "impossible":           # match scores of -32768, and some around the reach
            vp.msc[rng.random(vp.msc.shape) < 0.05] = -32768
            vp.msc[rng.random(vp.msc.shape) < 0.05] = -16385
            vp.msc[rng.random(vp.msc.shape) < 0.05] = -16384
        elif kind == "sticky_inserts":     # the offset may not be lowered
            vp.trans[5, ::3] = 0
            vp.trans[4, ::5] = -2
        elif kind == "loops":              # the entry score sinks fast
            vp.special[0] = vp.special[6] = -120
        elif kind == "entry":
            vp.trans[0, 1::2] -= 100
        elif kind == "far_moves":
            vp.trans[7, 9] = -17000
        elif kind == "low_base":
            vp.base = -9000
        else:                              # no positive match score
            vp.msc = np.minimum(vp.msc, -1).astype(np.int16)
    check(vps, database(vps[1], rng, 4000))


@pytest.mark.parametrize("top", [32767, 32766, 32765])
@pytest.mark.parametrize("M", [2, 70, 600, 1400])
def test_entry_score_at_the_top_of_the_range(M, top):
    """A match state that overflows in the first row, beside others that stay
    just below."""
    rng = np.random.default_rng(M + top)
    vp = synth.make_vit_profile(M, rng)
    vp.base = top
    vp.special[1] = 0
    vp.trans[0] = 0
    vp.msc[:] = -1
    vp.msc[3:, rng.integers(0, M, 1 + M // 20)] = 5      # residue codes below 3: no overflow in their row
    lengths = np.array([1, 1, 1, 2, 5, 40, 0, 300], dtype=np.uint32)
    offsets = np.concatenate([[0], np.cumsum(lengths[:-1], dtype=np.uint64)]).astype(np.uint64)
    res = rng.integers(0, 20, int(lengths.sum())).astype(np.uint8)
    res[:3] = [0, 5, 19]
    check([vp], synth.Database(residues=res, offsets=offsets, lengths=lengths))
