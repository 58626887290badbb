"""Tests of small batches once more with the one-launch step off. Up to some 32 rows the greedy and sampling steps take one launch, so that
these tests, as their own modules run them, say nothing about the streaming kernel with its per-row kernels and the class lists."""
import pytest

import _gpu_util
import test_gpu_fuzz
import test_gpu_odd_rows
import test_gpu_parity
import test_gpu_sample
from paper_2605_29986_b200 import binding as cz

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def two_launches(monkeypatch):
    as_it_is = _gpu_util.Ctx.__init__

    def without_one_launch(self, partitions):
        as_it_is(self, partitions)
        cz.cfgzip_set_tuning(self.h, "one_launch", 0)

    monkeypatch.setattr(_gpu_util.Ctx, "__init__", without_one_launch)


test_fused_tiny_shapes = test_gpu_parity.test_fused_tiny_shapes
test_fused_mixed_partitions = test_gpu_parity.test_fused_mixed_partitions_with_different_k
test_fused_degenerate_rows = test_gpu_parity.test_fused_degenerate_rows_and_status
test_fused_ties = test_gpu_parity.test_fused_ties_and_planted_spikes
test_fused_without_optional_outputs = test_gpu_parity.test_fused_without_optional_outputs_and_twice_for_determinism
test_fused_call_in_a_graph = test_gpu_parity.test_fused_call_can_be_captured_in_a_cuda_graph
test_steps_replayed_from_a_graph = test_gpu_parity.test_steps_replayed_from_a_cuda_graph_match_the_oracle
test_sample_tiny_shapes = test_gpu_sample.test_sample_tiny_shapes
test_sample_unaligned_rows = test_gpu_sample.test_sample_unaligned_rows_take_the_per_row_path
test_sample_mixed_partitions = test_gpu_sample.test_sample_mixed_partitions
test_sample_edge_rows = test_gpu_sample.test_sample_edge_rows_and_extreme_uniforms
test_sample_cold_distribution = test_gpu_sample.test_sample_cold_distribution_is_the_greedy_choice_and_t1_matches_the_greedy_lse
test_sample_unaligned_mixed = test_gpu_sample.test_sample_unaligned_rows_with_mixed_partitions
test_odd_rows_greedy = test_gpu_odd_rows.test_greedy
test_odd_rows_in_a_buffer = test_gpu_odd_rows.test_view_into_a_buffer
test_odd_rows_ties = test_gpu_odd_rows.test_ties_and_maxima_at_the_edges
test_odd_rows_mixed_partitions = test_gpu_odd_rows.test_mixed_partitions
test_odd_rows_sampling = test_gpu_odd_rows.test_sampling
test_host_step = test_gpu_odd_rows.test_host_step_with_pinned_buffers
test_random_shape = test_gpu_fuzz.test_random_shape
test_random_shape_sampling = test_gpu_fuzz.test_random_shape_sampling
