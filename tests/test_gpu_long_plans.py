"""Plans of long models that share the exact MSV kernel with other shared-memory sizes."""
import numpy as np
import pytest

from paper_1707_09683_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lengths", [(5000, 3500), (3500, 5000), (20000, 7000)])
def test_a_plan_launches_after_one_of_another_length_was_made(lengths):
    import torch

    import oracle
    from paper_1707_09683_gb300 import mpf

    rng = np.random.default_rng(3)
    recs = [synth.make_profile(M, rng) for M in lengths]
    dbh = synth.make_database(60, 200, 10, 600, rng)
    synth.plant_segments(dbh, recs, 0.3, rng)
    ctx = mpf.Context(0)
    db = mpf.Database(ctx, dbh.residues, dbh.offsets, dbh.lengths)
    profs = [mpf.Profile(ctx, r) for r in recs]
    outs = [[torch.zeros(db.n_seqs, dtype=t, device="cuda") for t in (torch.uint8, torch.uint8, torch.float32)]
            for _ in recs]
    plans = [mpf.Plan(ctx, mpf.MSV, [p], db, *o) for p, o in zip(profs, outs)]
    for plan in plans:
        plan.launch()
    ctx.sync()
    for r, o in zip(recs, outs):
        for got, want in zip(o, oracle.msv(r, dbh.residues, dbh.offsets, dbh.lengths)):
            np.testing.assert_array_equal(got.cpu().numpy(), want)
    for plan in plans:
        plan.close()
