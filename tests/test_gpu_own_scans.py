"""The parity tests of the plain scans on each method's own kernels."""
from tests.pinned_plans import own_scans  # noqa: F401
from tests.test_gpu_acv import (  # noqa: F401
    pytestmark, test_acv_capacity_short_and_device_api, test_acv_edges, test_acv_est_text,
    test_acv_many_patterns_per_position_overflow, test_acv_random_sets, test_wmv_est_text_and_overflow,
    test_wmv_random_sets)
from tests.test_gpu_parity import (  # noqa: F401
    est_text_full, test_ac_random_small, test_device_api_capacity_and_status, test_edge_cases,
    test_est_sets_on_64mib_prefix, test_every_position_matches_overflow_path, test_large_sets_full_text,
    test_pfac_est_sets_and_every_position_matching, test_pfac_random_small, test_scan_to_host_in_pieces,
    test_scan_to_host_pinned_buffers_and_capacity, test_small_uniform_workload, test_unaligned_device_text,
    test_wm_byte_path_groups_and_overflow, test_wm_random_small)
