"""The tuner runs every set of kernels once: settings that only rename the
direct pass (force modes 2, 3 and 5, lanes per particle) share its time, and
the choice it saves carries the pass's own name."""
import pytest

from paper_2002_03120_gb300 import autotune


@pytest.mark.parametrize("precision", [0, 1])
def test_aliases_are_timed_once_and_never_chosen(precision):
    runs = []

    def noisy(setting):   # every later run of the direct pass happens to be faster
        runs.append(setting)
        return 100.0 + 10.0 * (setting["newton3"] in (1, 4)) - 0.01 * len(runs)

    best, table = autotune.search(autotune.once_per_kernel(noisy), precision=precision)
    kernels = {(r["newton3"] in (1, 4), r["skin"], r["block"], r["cells"]) for r in table}
    assert len(runs) == len(kernels) < len(table)
    assert best["newton3"] == 0 and best["tpp"] == 1
