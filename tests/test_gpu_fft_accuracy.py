"""Error of whole calls against 64 bits on grids with a factor 3, no larger than with the radix plans that these
lengths had before theirs of 24 elements a thread: the limits are what those measured on the same inputs."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,seed,limit", [
    ("run_scan_192x96", 1, 2.261e-6), ("run_scan_192x96", 2, 2.178e-6), ("run_scan_192x96", 3, 2.203e-6),
    ("propagate_scan_384", 1, 1.824e-6), ("propagate_scan_384", 2, 2.577e-6), ("propagate_scan_384", 3, 2.416e-6)])
def test_error_against_64_bits(name, seed, limit):
    import __graft_entry__
    __graft_entry__.build()
    from perf import cases
    case = next(c for c in cases.listed() if c["name"] == name)
    out, ref = cases.run(cases.prepare(case, seed)), cases.exact(case, seed)
    assert float((out - ref).norm() / ref.norm()) <= limit
