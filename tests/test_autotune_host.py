"""Host logic of the autotuner on a fake of the binding (no GPU)."""
import types

import pytest

pytest.importorskip("torch")

from paper_1610_07522_gb300 import autotune as A
from paper_1610_07522_gb300 import binding as B


@pytest.mark.parametrize("fused", [1, 0, None])
def test_tune_box_times_line_shapes_on_the_passes_that_use_them(monkeypatch, fused):
    """The line passes' block shapes are timed while h psi takes them (general
    passes); the choice of passes is afterwards what it was.  None: a context
    that has no fused passes."""
    knobs = {k: v[0] for k, v in A.CANDIDATES.items()}
    knobs[B.SKY_KNOB_FUSED_H] = fused or 0
    seen = []

    def tune_set(ctx, knob, value):
        if knob == B.SKY_KNOB_FUSED_H and value == 1 and fused is None:
            raise B.SkyError(B.SKY_EINVAL, "no fused passes")
        knobs[knob] = value

    monkeypatch.setattr(A.B, "sky_tune_set", tune_set)
    monkeypatch.setattr(A.B, "sky_tune_get", lambda ctx, knob: knobs[knob])
    monkeypatch.setattr(A.B, "sky_apply_h", lambda *a: seen.append(knobs[B.SKY_KNOB_FUSED_H]))
    monkeypatch.setattr(A.B, "sky_overlap", lambda *a: None)
    monkeypatch.setattr(A, "_key", lambda s: "box")
    monkeypatch.setattr(A, "_time", lambda fn, stream, reps: fn() or 1.0)
    monkeypatch.setattr(A.torch.cuda, "synchronize", lambda *a: None)
    pair = [None, None]
    box = types.SimpleNamespace(ctx=None, stream=None, I=(4, 2), prec=B.SKY_F32, device=0, U=pair, Bf=pair,
                                W=pair, psi=pair, h=pair, H=pair)
    A.tune_box(box)
    assert len(seen) == len(A.CANDIDATES[B.SKY_KNOB_LINE_YZ]) + len(A.CANDIDATES[B.SKY_KNOB_LINE_X])
    assert set(seen) == {0}
    assert knobs[B.SKY_KNOB_FUSED_H] == (fused or 0)
