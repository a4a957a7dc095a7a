"""A tune-cache line of other kernels (an earlier revision, or none in its key)
does not decide a plan's variant; the line of the plan's own kernels does."""
import re

import gen
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [32, 72])
def test_lines_of_other_kernels_do_not_count(n, monkeypatch, tmp_path):
    import paper_2110_07670_gb300 as ace
    cache = tmp_path / "tune"
    monkeypatch.setenv("ACE_TUNE_CACHE", str(cache))
    monkeypatch.delenv("ACE_ROW_BLOCK", raising=False)
    args = ((n, n, n), gen.cubic_cell(10.0), 30.0, 4, "mixed")
    ace.Plan(*args).close()
    key = cache.read_text().splitlines()[-1].split(" = ")[0]
    head, rev = re.fullmatch(r"(.* sm\d+) k(\d+)", key).groups()
    cache.write_text(f"{head} = 1 1 0 0\n{head} k{int(rev) - 1} = 1 1 0 0\n")
    plan = ace.Plan(*args)
    assert not plan.config()["from_tune_cache"]
    plan.close()
    cache.write_text(f"{key} = 1 1 0 0\n{head} k{int(rev) - 1} = 4 2 0 0\n")
    plan = ace.Plan(*args)
    cfg = plan.config()
    assert cfg["from_tune_cache"] and (cfg["pair_variant"], cfg["pair_streams"]) == (1, 1)
    plan.close()
