"""The smoke run launches every persistent kernel and the tensor path."""
import pytest

import paper_1905_00689_gb300 as package

pytestmark = pytest.mark.gpu


def test_smoke_runs_every_persistent_kernel(cuda_device, monkeypatch):
    import __graft_entry__
    seen = set()

    class Recording(package.LSTMApprox):
        def close(self):
            if getattr(self, "h", None):
                seen.add((self.query(package.Q_LAST_PATH), self.query(package.Q_PERSISTENT_VARIANT)))
            super().close()

    monkeypatch.setattr(package, "LSTMApprox", Recording)
    __graft_entry__.smoke()
    assert {v for path, v in seen if path == package.PATH_PERSISTENT} == {1, 2, 3}
    assert package.PATH_TENSOR in {path for path, _ in seen}
