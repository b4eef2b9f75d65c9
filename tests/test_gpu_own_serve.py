"""The server's tests with requests that run in the transition-table kernel."""
from tests.pinned_plans import own_scans  # noqa: F401
from tests.test_gpu_serve import (  # noqa: F401
    base, pytestmark, sets, test_large_requests_split_or_plain, test_results_alone_and_in_the_mix,
    test_short_estimate_reruns_with_exact_capacity, test_tight_budget_admission_waits)
