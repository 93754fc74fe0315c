"""HeMult.check reads every flag that a run's bounded waits can set: all its plans and parameter sets, each
cleared even where an earlier one had expired (library calls faked; no GPU)."""
import types

import pytest

from paper_2501_07047_gb300 import hefx
from paper_2501_07047_gb300.hemult import HeMult


def he_mult(modup, plans):
    hm = object.__new__(HeMult)
    hm.ctx, hm.modup, hm.plans = 1, modup, plans
    hm.plan_pq, hm.pQ, hm.pQr, hm.pQP = "pq", "Q", "Qr", "QP"
    hm.torch = types.SimpleNamespace(cuda=types.SimpleNamespace(current_stream=lambda: "current"))
    return hm


@pytest.mark.parametrize("modup,plans", [("up", []), (None, [(None, "a"), ("b", "c")])])
@pytest.mark.parametrize("expired", [set(), {"pq"}, {"up", "a", "QP"}, {"Q"}])
def test_every_flag_is_read(monkeypatch, modup, plans, expired):
    asked = []

    def fake(kind):
        def check(ctx, handle, stream=None):
            assert ctx == 1 and stream == "current"
            asked.append((kind, handle))
            if handle in expired:
                raise hefx.HefxError(hefx.HEFX_ETIMEOUT, str(handle))
        return check

    for kind in ("modup", "bconv", "stream"):
        monkeypatch.setattr(hefx, f"hefx_{kind}_check", fake(kind))
    want = ([("modup", "up")] if modup else []) + [("bconv", p) for pair in plans for p in pair if p]
    want += [("bconv", "pq"), ("stream", "Q"), ("stream", "Qr"), ("stream", "QP")]
    hm = he_mult(modup, plans)
    if expired & {h for _, h in want}:
        with pytest.raises(hefx.HefxError) as e:
            hm.check()
        assert e.value.status == hefx.HEFX_ETIMEOUT
    else:
        hm.check()
    assert asked == want


def test_other_errors_are_not_held_back(monkeypatch):
    def check(ctx, handle, stream=None):
        raise hefx.HefxError(hefx.HEFX_EINVAL, "closed")

    monkeypatch.setattr(hefx, "hefx_bconv_check", check)
    with pytest.raises(hefx.HefxError) as e:
        he_mult(None, []).check()
    assert e.value.status == hefx.HEFX_EINVAL
