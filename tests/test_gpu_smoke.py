"""The smoke run reaches the solver's main paths, not only its smallest one."""
import pytest

import __graft_entry__ as entry
from paper_2302_12199_gb300 import mst

pytestmark = pytest.mark.gpu


def test_smoke_reaches_the_main_paths(monkeypatch):
    launched = set()

    class Counted(mst.Solver):
        def __init__(self, *args, **kw):
            super().__init__(*args, **kw)
            self.profile(True, classes=[])

        def close(self):
            if getattr(self, "h", None):
                launched.update(k for k, v in self.profile_stats().items() if v[0])
            super().close()
    monkeypatch.setattr(mst, "Solver", Counted)
    entry.smoke()
    assert launched >= {"base", "min_edges", "graph", "pivot", "partition", "jump", "filter", "finalize"}
