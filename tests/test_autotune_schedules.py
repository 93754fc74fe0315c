"""The tuner can choose the cluster schedule wherever the library's own choice is another one (timings faked;
no GPU), and a choice that was cached is applied without timing again."""
import pytest

from paper_2501_07047_gb300 import autotune


@pytest.mark.parametrize("logn", [14, 15, 17])
@pytest.mark.parametrize("cluster_ms,want", [(0.9, ("cudacore", 1, 0, 0)), (1.1, ("cudacore", 0, 0, 0))])
def test_cluster_schedule_can_win(monkeypatch, tmp_path, logn, cluster_ms, want):
    import torch
    monkeypatch.setattr(autotune, "CACHE", str(tmp_path / "tune.json"))
    monkeypatch.setattr(torch.cuda, "get_device_name", lambda *a: "FAKE-GPU")
    timed, applied = [], []

    def times(ctx, params, logn, primes, batch=4, reps=5, cands=None):
        timed.append(cands)
        ms = {("cudacore", 0, 0, 0): 1.0, ("cudacore", 1, 0, 0): cluster_ms}
        return {autotune.key_of(c): ms.get(c, 2.0) for c in (autotune.candidates(logn) if cands is None else cands)}

    monkeypatch.setattr(autotune, "time_candidates", times)
    monkeypatch.setattr(autotune, "apply", lambda ctx, p, cand: applied.append(cand))
    for _ in range(2):
        assert autotune.tune(None, None, logn, [268042241]) == "cudacore"
    assert applied == [want, want] and timed == [None, [("cudacore", 1, 0, 0)]]


@pytest.mark.parametrize("cand,schedule", [(("tensor", 7, 0, 64), "auto"), (("cudacore", 0, 0, 0), "auto"),
                                           (("cudacore", 1, 0, 0), "cluster"), (("cudacore", 2, 0, 0), "two_pass")])
def test_apply_leaves_no_schedule_behind(monkeypatch, cand, schedule):
    """The schedule that was timed last does not stay where another configuration is applied."""
    calls = {}
    monkeypatch.setattr(autotune.hefx, "hefx_params_set_cc_schedule", lambda c, p, s: calls.update(schedule=s))
    monkeypatch.setattr(autotune.hefx, "hefx_params_set_tensor_config", lambda *a: calls.update(split=a[2:]))
    monkeypatch.setattr(autotune.hefx, "hefx_params_set_auto_path", lambda p, path: calls.update(path=path))
    autotune.apply(1, 2, cand)
    assert calls["schedule"] == schedule and calls["path"] == cand[0] and ("split" in calls) == (cand[0] == "tensor")


def test_no_alternatives_elsewhere():
    assert [n for n in range(3, 18) if autotune.alternatives(n)] == [14, 15, 17]
