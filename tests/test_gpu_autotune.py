"""The batch autotuner: its cache file and what it times."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _batch(h_max=3.0):
    import paper_2405_14551_gb300.lbcg as L
    from paper_2405_14551_gb300 import workloads as W
    runs = [W.Workload(f"r{k}", (24 + 8 * k, 24, 16), 0, dict(W.BASE, A_h=0.1, h_max=h_max), 4,
                       centres=np.array([[12.0, 12.0, 8.0]]), radii=np.array([5.0])) for k in range(3)]
    return L.Batch(runs)


def test_entries_of_another_revision_are_not_used(tmp_path, monkeypatch):
    """A line without this build's revision, as builds with other tile shapes wrote
    it, is passed over; the line written here is used."""
    path = tmp_path / "tune.txt"
    monkeypatch.setenv("LBCG_TUNE_CACHE", str(path))
    assert _batch().autotune(steps=1)[3] == 0
    key, tile, bps, ms = path.read_text().split()
    assert _batch().autotune(steps=1)[3] == 1
    revision, _, rest = key.partition("|")
    assert revision.startswith("rev")
    for old in (rest, f"rev0|{rest}"):
        path.write_text(f"{old} 3 1 0.000001\n")
        _, _, t, cached = _batch().autotune(steps=1)
        assert cached == 0 and t > 1e-5


@pytest.mark.parametrize("h_max,shapes", [(3.0, 3), (5.0, 1)])
def test_each_shape_is_timed_once(tmp_path, monkeypatch, h_max, shapes):
    """Indexes that launch the same shape are timed once: per shape and number of
    CTAs an SM two warm-up steps and one timed, of two launches each; one step more
    for each run that has not begun."""
    import paper_2405_14551_gb300.lbcg as L
    monkeypatch.setenv("LBCG_TUNE_CACHE", str(tmp_path / "tune.txt"))
    b = _batch(h_max)
    before = L.lb_launch_count()
    b.autotune(steps=1, use_cache=False)
    assert L.lb_launch_count() - before == 2 * 3 + shapes * 3 * 3 * 2
