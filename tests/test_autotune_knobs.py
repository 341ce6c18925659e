"""The tuner tries only settings that act on what it times: cc_batch_* calls do not
read batch_small_n (the sizes and the number of the jobs decide), and heavy lists
above 2048 vertices are never looked at inside the barrier, so larger limits are one
setting.  A choice stored with batch_small_n by an earlier tuner is not carried over
to the servers of the process."""
import pytest

from paper_1507_05086_gb300 import autotune


class FakeGraph:
    n, nnz, max_degree = 5000, 60_000, 40


def test_batch_knobs_act_on_batches():
    assert "batch_small_n" not in autotune.BATCH_KNOBS


def test_inline_heavy_candidates_differ():
    cc = pytest.importorskip("paper_1507_05086_gb300")
    limits = [min(v, 2048) for v in autotune.ROUND_KNOBS["inline_heavy"]]
    assert len(set(limits)) == len(limits)
    default = cc.default_tuning().to_dict()["inline_heavy"]
    assert default == 2048 and default in autotune.ROUND_KNOBS["inline_heavy"]


def test_stored_choice_applies_its_own_knobs_only(tmp_path, monkeypatch):
    pytest.importorskip("paper_1507_05086_gb300")
    path = str(tmp_path / "tuning.json")
    graphs = [FakeGraph()] * 3
    applied = []
    monkeypatch.setattr(autotune, "device_key", lambda: "dev")
    monkeypatch.setattr(autotune.native, "set_batch_tuning", lambda t: applied.append(dict(t)))
    autotune.store(path, "dev", "batch", autotune.batch_class(graphs),
                   {"tuning": {"batch_team_blocks": 16, "batch_small_n": 1 << 14}, "ms": 1.0})
    base = autotune.native.default_tuning().to_dict()
    hit = autotune.tune_batch(graphs, cache=path)
    assert hit["source"] == "cache" and hit["tuning"] == {"batch_team_blocks": 16}
    assert applied == [dict(base, batch_team_blocks=16)]
    # asked for by name, it is applied
    hit = autotune.tune_batch(graphs, cache=path, knobs={"batch_small_n": (1 << 14, 1 << 16)})
    assert applied[-1] == dict(base, batch_small_n=1 << 14)
