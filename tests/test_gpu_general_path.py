"""The tests of small problems, on the general path.

eta_decode takes small problems in one kernel, so tests whose sizes are small reach that kernel and none of the three of the general
path, whose edges (tiles, passes and segments of the screening, rescue windows, set-up of the streaming kernel, queued
launches, what is left in the scratch) several of them are about.  Here they run once more with a build of the same sources that
takes the general path whatever the size."""
import pytest

from tests.test_gpu_back_to_back import (test_captured_calibration_bounds_and_staged_query, test_queued_bounds_between_append_and_step,  # noqa: F401
                                         test_queued_calibrations_share_a_scratch, test_queued_steps_equal_separate_steps,
                                         test_queued_steps_fetch_their_queries_into_one_buffer,
                                         test_thresholds_written_where_the_step_before_left_its_output)
from tests.test_gpu_full_configs import test_c1_tiny_16_decode_steps  # noqa: F401
from tests.test_gpu_giveup import test_a_wait_that_runs_out_reports_timeout_and_leaves_the_workspace_usable  # noqa: F401
from tests.test_gpu_packed import (test_decode_on_packed_summaries_matches_the_oracle,  # noqa: F401
                                   test_packed_screen_for_other_group_sizes_and_the_bound_diagnostic)
from tests.test_gpu_paged import test_paged_cache_equals_contiguous_bit_for_bit  # noqa: F401
from tests.test_gpu_parity import (test_chained_gpu_path_and_multi_step_append, test_decode_matches_oracle_on_scaled_configs,  # noqa: F401
                                   test_edge_shapes_and_group_sizes, test_frozen_constants_against_predicted_mode_on_the_same_cache,
                                   test_minus_infinite_threshold_and_dense_flag_are_softmax_attention,
                                   test_plus_infinite_threshold_attends_rescue_pins_and_tail_only,
                                   test_query_magnitudes_outside_the_fp16_range_screen_like_their_scaled_twins,
                                   test_query_staged_from_pinned_memory_and_output_written_to_it,
                                   test_rescue_window_longer_than_four_segments_and_many_segment_counts, test_run_to_run_determinism,
                                   test_sphere_term_binds_and_large_logits_stay_finite, test_strided_cache_layout_bthd,
                                   test_threshold_equal_to_a_bound_admits_the_block_on_the_device, test_ungated_newest_token)
from tests.test_gpu_random_sweep import test_random_configuration_matches_the_oracle  # noqa: F401
from tests.test_gpu_rescue_window import test_long_windows_match_the_oracle  # noqa: F401
from tests.test_gpu_screen_tiles import test_selection_matches_the_rule  # noqa: F401
from tests.test_zz_no_alloc import (test_scratch_left_by_a_different_call_is_never_consumed,  # noqa: F401
                                    test_static_scratch_variant_matches_eta_decode_twice_in_a_row)

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def general_path(monkeypatch):
    from paper_2609_20888_b200 import binding as eb
    from paper_2609_20888_b200 import build as ebuild
    ebuild.build()
    eb.load()
    monkeypatch.setattr(eb, "_lib", eb.load(ebuild.build_general_variant()))
    assert eb.eta_decode_launches(eb.CacheDesc(1, 4, 1, 128, 64, 128, 2, 0, 0, 128, 0, 0, 128), eb.DecodeParams()) == 3
