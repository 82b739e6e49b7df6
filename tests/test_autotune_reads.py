"""The autotuner spends no trials on options that the configuration's solves do
not read."""
import pytest

from paper_2302_12199_gb300.autotune import (QUANTILE_CANDIDATES, READ_BY, RELABEL_SHAPE_CANDIDATES, SHAPE_CANDIDATES,
                                             autotune, label)


@pytest.mark.parametrize("classes,stages", [
    ({"base"}, set()),                                                    # one block per graph
    ({"min_edges", "graph", "finalize"}, set()),                          # plain rounds in one launch
    ({"pivot", "partition", "filter", "jump", "graph"}, {"quantile", "shape"}),   # planned Filter-Boruvka
    ({"min_edges", "hook", "jump", "relabel_min"}, {"shape", "relabel"}),  # rounds driven by the host
    ({"min_edges", "hook", "jump", "dedupe"}, {"shape", "relabel"}),
])
def test_stages_that_nothing_reads_are_skipped(classes, stages):
    tried = []

    def trial(cfg):
        tried.append(dict(cfg))
        return 1.0
    base = dict(variant="filter")
    best, res = autotune(trial, [base], reps=1, relabel_shapes=RELABEL_SHAPE_CANDIDATES, launched=lambda cfg: classes)
    assert best == base
    got = {s for cfg in tried for s, k in (("quantile", "pivot_quantile"), ("shape", "block_threads"),
                                           ("relabel", "relabel_block_threads")) if k in cfg}
    assert got == stages
    assert len(res) == 1 + 3 * ("quantile" in stages) + 8 * ("shape" in stages) + 8 * ("relabel" in stages)


def test_every_later_option_names_its_readers():
    from paper_2302_12199_gb300.mst import KERNEL_CLASSES
    for c in QUANTILE_CANDIDATES + SHAPE_CANDIDATES + RELABEL_SHAPE_CANDIDATES:
        assert all(READ_BY[k] and set(READ_BY[k]) <= set(KERNEL_CLASSES) for k in c), label(c)
