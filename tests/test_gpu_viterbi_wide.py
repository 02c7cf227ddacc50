"""The 32-bit Viterbi kernels at the shapes that their tests name.

Realistic profiles have a uniform entry move, with which the packed kernel
takes them; here one node's entry move is lower, so the same tests run the
kernels of their docstrings (teams, one warp per sequence, rows in device
memory).
"""
import pytest

from paper_1707_09683_gb300 import synth
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
