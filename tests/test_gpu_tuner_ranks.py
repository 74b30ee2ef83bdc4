"""GPU: the autotuner measures the solve's schedule and staging only at the ranks whose
sweeps have them, and does not take choices cached for earlier candidates."""
import pytest

from paper_2311_00921_gb300 import hss
from paper_2311_00921_gb300 import inputs as I

pytestmark = pytest.mark.gpu

ALL = {f"{s}/{g}" for s in ("async", "levels") for g in ("largest_panels", "fewest_waves")}
ONE = {"async/largest_panels"}


@pytest.mark.parametrize("prec,rank,measured", [
    ("fp64", 16, ALL), ("fp64", 17, ONE), ("fp32", 32, ALL), ("fp32", 33, ONE)])
def test_candidates_follow_the_rank(prec, rank, measured):
    dev = hss.HSS(I.random_hss(3, 64, rank, seed=rank, orthonormal=False))
    t = dev.tune(prec, nrhs=2)
    assert set(t["measured"]["solve_ms"]) == measured
    assert t["schedule"] == "async" or measured == ALL
    assert t["staging"] == "largest_panels" or measured == ALL


def test_cached_choice_of_earlier_candidates_is_measured_again(tmp_path):
    h = I.random_hss(2, 64, 20, seed=1, orthonormal=False)
    cache = tmp_path / "tune.txt"
    hss.HSS(h).tune("fp64", nrhs=2, cache=str(cache))
    version, rest = cache.read_text().split(" ", 1)
    assert version.startswith("v") and version[1:].isdigit()
    for old in (rest, f"v{int(version[1:]) - 1} {rest}"):
        cache.write_text(old)
        assert not hss.HSS(h).tune("fp64", nrhs=2, cache=str(cache))["from_cache"]
        assert hss.HSS(h).tune("fp64", nrhs=2, cache=str(cache))["from_cache"]
