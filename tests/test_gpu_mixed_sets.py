"""Plans whose shorter queries share warps in mixed sets (bit-exact against the oracle).

Queries of the default configuration and fewer than 32 lanes each get as many
lanes of a warp as their nodes need: sets that fill the warp and sets that do
not, groups of one lane, ragged last lanes, strong profiles (overflow, J
chaining and its rescoring launch), per-code best scores for sequences whose
cells never rise, long sequences in segments, and a database with higher
residue codes, where no mixed set is formed.
"""
import numpy as np
import pytest

from paper_1707_09683_gb300 import synth

pytestmark = pytest.mark.gpu

BATCHES = {
    "sweep": [48, 100, 200, 400, 800, 1600],
    "short": [1, 7, 30, 33, 49, 50, 64, 77, 97],
    "ragged": [1279, 1100, 640, 333, 334, 335, 65, 129, 960, 1, 47],
    "two": [120, 1200],
}


@pytest.mark.parametrize("codes", [20, 21])
@pytest.mark.parametrize("strong", [False, True])
@pytest.mark.parametrize("batch", list(BATCHES))
def test_mixed_sets(batch, strong, codes):
    import torch

    import oracle
    from paper_1707_09683_gb300 import mpf

    rng = np.random.default_rng(len(batch) + 10 * strong + codes)
    if strong:
        recs = [synth.random_profile(M, 20, rng, cost_hi=26, bias=20, base=190, tbm=10, tec=3, tjb=8)
                for M in BATCHES[batch]]
    else:
        recs = [synth.make_profile(M, rng) for M in BATCHES[batch]]
    lengths = np.concatenate([rng.integers(0, 400, 300), [9000, 3000, 0, 1, 2, 3, 4, 5]]).astype(np.uint32)
    offsets = np.concatenate([[0], np.cumsum(lengths[:-1], dtype=np.uint64)]).astype(np.uint64)
    res = synth.draw_residues(int(lengths.sum()), rng)
    res[-1] = codes - 1
    ctx = mpf.Context(0)
    db = mpf.Database(ctx, res, offsets, lengths)
    profs = [mpf.Profile(ctx, r) for r in recs]
    n, q = lengths.size, len(profs)
    want = [[f(r, res, offsets, lengths, nthreads=16) for r in recs] for f in (oracle.msv, oracle.ssv)]
    for filt in (mpf.MSV, mpf.SSV, mpf.MSV_SSV):
        blocks = want if filt == mpf.MSV_SSV else [want[filt]]
        out = [torch.full((len(blocks) * q * n,), 99, dtype=t, device="cuda")
               for t in (torch.uint8, torch.uint8, torch.float32)]
        plan = mpf.Plan(ctx, filt, profs, db, *out)
        assert sum(g["n_queries"] for g in plan.groups()) == q
        if codes == 20:
            assert any(g["queries_per_warp"] > 1 for g in plan.groups())
        plan.launch()
        ctx.sync()
        for j in range(3):
            exp = np.concatenate([w[j] for b in blocks for w in b])
            np.testing.assert_array_equal(out[j].cpu().numpy(), exp, err_msg=f"filter {filt} output {j}")
