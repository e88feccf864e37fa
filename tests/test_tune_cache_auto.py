"""The launch-shape file holds the default form of the levels above the tail (sweep -1); host only, no GPU."""
import pytest


@pytest.fixture(scope="module")
def hn():
    import __graft_entry__ as g
    g.build()
    from paper_0904_4152_gb300 import hn
    return hn


def test_the_default_form_is_stored_and_found(hn, tmp_path):
    path = str(tmp_path / "tune.txt")
    shape = (5, 16, 2, 0, 1, 0, 0, -1)
    hn.hn_tune_cache_store(path, "GPU", 10, 1, 0, 0, 2, shape)
    assert hn.hn_tune_cache_lookup(path, "GPU", 10, 1, 0, 0, 2) == shape
    with pytest.raises(hn.HnError) as e:
        hn.hn_tune_cache_store(path, "GPU", 10, 1, 0, 0, 2, shape[:7] + (-2,))
    assert e.value.status == hn.HN_ERR_ARG
