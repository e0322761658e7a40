"""PCAPreprocessor.fit reports a fit whose device-side wait ran out instead of keeping its outputs."""
import pytest
import torch


def test_fit_raises_on_timeout(monkeypatch):
    from paper_2602_01330_gb300 import dualk
    from paper_2602_01330_gb300.preprocess import PCAPreprocessor

    class Ctx:
        error = None

        def sync_status(self, stream=None):
            if self.error:
                raise self.error

    monkeypatch.setattr(dualk, "pca_fit", lambda ctx, x, k, sweeps: {"k": k})
    monkeypatch.setattr(torch.cuda, "is_current_stream_capturing", lambda: False)
    ctx = Ctx()
    assert PCAPreprocessor(ctx).fit(torch.zeros(4, 3)).model == {"k": 3}
    ctx.error = RuntimeError("device-side wait exceeded its bound")
    pre = PCAPreprocessor(ctx)
    with pytest.raises(RuntimeError):
        pre.fit(torch.zeros(4, 3))
    assert pre.model is None
    # nothing has run yet inside a capture: the check is the caller's
    monkeypatch.setattr(torch.cuda, "is_current_stream_capturing", lambda: True)
    assert pre.fit(torch.zeros(4, 3)).model == {"k": 3}
