"""The autotuner starts from the library's own defaults and tries each of them."""
import os
import re

from paper_2506_06269_gb300 import tune

CSRC = os.path.join(os.path.dirname(os.path.abspath(tune.__file__)), "csrc")


def _constant(file, name):
    with open(os.path.join(CSRC, file)) as f:
        m = re.search(r"\b%s = ([0-9.]+)f?\b" % name, f.read())
    return float(m.group(1))


def test_defaults_are_the_library_defaults():
    d = tune.DEFAULTS
    assert d["pair_per_round"] == _constant("sidm_pairs.cu", "kPerRoundDefault")
    assert d["knn_groups"] == _constant("sidm_knn.cu", "kGroupsDefault")
    assert d["knn_chains"] == _constant("sidm_knn.cu", "kChainsDefault")
    assert d["knn_batch"] == _constant("sidm_knn.cu", "kBatchDefault")
    assert d["knn_flush"] == _constant("sidm_knn.cu", "kFlushNodeDefault")
    assert abs(d["knn_slack"] - _constant("sidm_knn.cu", "kGuessSlackDefault")) < 1e-6
    for knobs in (tune.KNN_KNOBS, tune.PAIR_KNOBS):
        for name, values in knobs.items():
            assert d[name] in values, name
