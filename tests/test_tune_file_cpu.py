"""The tuning file and the lists of variants: a measured line counts only for the list of
variants it was measured with."""
import pytest


@pytest.fixture
def query(tmp_path):
    from paper_1305_6653_gb300 import fde_tune_cache, fde_tune_query

    def load(text):
        f = tmp_path / "t.txt"
        f.write_text(text)
        fde_tune_cache(str(f))
        return fde_tune_query
    yield load
    fde_tune_cache(None)


def test_lines_of_another_list_are_measured_again(query):
    # as written before the lists changed: 384 x 8 rows / the shared-memory ring, 512 threads a row
    q = query("trsv 1 1024 33 1 3 # 0.1510 0.1455 0.1602 0.1449 ms\nmatvec 0 2048 256 0 1 # 0.1904 0.1850 0.1911 ms\n"
              "trsv 1 2048 129 1 2 # list 1: 0.1 0.2 0.3 0.4 ms\n")
    assert q(1, 1024, 33, "fp32") == q(0, 2048, 256, "fp64") == q(1, 2048, 129, "fp32") == -1


def test_lines_of_this_list_and_lines_by_hand_count(query):
    q = query("trsv 1 1024 33 1 3 # list 2: 0.1510 0.1455 0.1602 0.1449 ms\nmatvec 0 2048 256 0 1\n")
    assert q(1, 1024, 33, "fp32") == 3 and q(0, 2048, 256, "fp64") == 1
