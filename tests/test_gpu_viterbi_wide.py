"""The 32-bit Viterbi kernels at the shapes that their tests name.

Realistic profiles have a uniform entry move, with which the packed kernel
takes them; here one node's entry move is lower, so the same tests run the
kernels of their docstrings (teams, one warp per sequence, rows in device
memory).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_1707_09683_gb300 import mpf, synth
from test_gpu_viterbi import (ctx, test_largest_model, test_long_model, test_long_segment_variants,  # noqa: F401
                              test_msv_to_viterbi_stage, test_multi_query_launch, test_realistic_profiles)
from test_gpu_viterbi_long import (test_device_rows_below_striped_length, test_longest_model,  # noqa: F401
                                   test_mixed_groups_in_one_call, test_more_groups_than_fork_streams,
                                   test_msv_to_viterbi_stage_long_model, test_realistic_long_profiles)
from test_gpu_viterbi_team import (test_dual_launch_splits_queries_by_survivors, test_one_warp_kernel_many_sequences,  # noqa: F401
                                   test_team_lengths, test_team_mixed_with_other_kernels, test_team_pass_fractions,
                                   test_team_short_sequences)

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def one_entry_move_lower(monkeypatch):
    uniform = synth.make_vit_profile

    def make(M, rng):
        v = uniform(M, rng)
        v.trans[0, M // 2] -= 3
        return v
    monkeypatch.setattr(synth, "make_vit_profile", make)


def test_scan_without_room_for_the_packed_kernels_lists(ctx):
    """The packed kernel lists the sequences that it leaves to the 32-bit
    kernels (4 bytes per sequence and query); where that memory is not there,
    the 32-bit kernels score the queries."""
    rng = np.random.default_rng(31)
    n, q = 500_000, 60
    dbh = synth.Database(residues=rng.integers(0, 20, n, dtype=np.uint8), offsets=np.arange(n, dtype=np.uint64),
                         lengths=np.ones(n, np.uint32))
    db = mpf.Database(ctx, dbh.residues, dbh.offsets, dbh.lengths)
    rec = synth.make_vit_profile(50, rng)
    rec.trans[0] = rec.trans[0, 0]          # packed, if there is room
    vp = mpf.VitProfile(ctx, rec)
    out = [torch.zeros(q * n, dtype=t, device="cuda") for t in (torch.int16, torch.uint8, torch.float32)]
    ctx.sync()
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info(0)
    hold = torch.empty(free - (96 << 20), dtype=torch.uint8, device="cuda")
    try:
        mpf.viterbi_scan(ctx, [vp] * q, db, *out)
        ctx.sync()
    finally:
        del hold
        torch.cuda.empty_cache()
    for got, want in zip(out, oracle.viterbi(rec, dbh.residues, dbh.offsets, dbh.lengths, nthreads=16)):
        want = torch.from_numpy(want).cuda()
        assert all(torch.equal(got[i * n:(i + 1) * n], want) for i in range(q))
    vp.close()
    db.close()
