"""Saved autotuner tables name the version of the launch shapes their numbers index; host code, no GPU."""
import pytest

HOP = "hop prec=1 recon=12 dagger=0 epi=0 red=0 full=0 lat=2x2x2x2 n5=7"


@pytest.fixture
def api():
    from paper_1512_03487_gb300 import api
    yield api
    api.lqcd_tune_clear()


def _table(api, path):
    api.lqcd_tune_save(str(path))
    return {ln.split("\t")[1]: ln.split("\t") for ln in path.read_text().splitlines()}


def test_saved_hop_choices_carry_the_version_of_the_shapes(api, tmp_path):
    api.lqcd_tune_clear()
    path = tmp_path / "table.txt"
    path.write_text(f"4\t{HOP}\n3\thost-test-other\n")  # written by hand: taken as it is
    api.lqcd_tune_load(str(path))
    assert api.lqcd_tune_get(HOP) == 4
    lines = _table(api, path)
    assert lines["host-test-other"] == ["3", "host-test-other"]
    value, _, tag = lines[HOP]
    assert value == "4" and tag.startswith("shapes=")
    api.lqcd_tune_clear()
    api.lqcd_tune_load(str(path))  # what was saved comes back
    assert api.lqcd_tune_get(HOP) == 4 and api.lqcd_tune_entries() == 2
    assert _table(api, path) == lines
    api.lqcd_tune_clear()
    other = f"shapes={int(tag[7:]) + 1}"
    for wrong in (other, "shapes=1", "shapes=", "", tag + "0"):
        path.write_text(f"4\t{HOP}\t{wrong}\n5\thost-test-other\n")
        api.lqcd_tune_load(str(path))  # numbers of another list: the hop is timed again, the rest is taken
        assert api.lqcd_tune_get(HOP) == -1 and api.lqcd_tune_get("host-test-other") == 5
