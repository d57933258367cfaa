"""The autotuner's cache file belongs to the parameters it was tuned for: a table
of another context of the same sizes, whose primes take other kernels, or of a
file whose key does not name the primes, is not loaded."""
import json

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2507_04775_gb300 import Context, find_primes  # noqa: E402


def context(bits):
    q = find_primes(14, bits, 4)
    return Context(14, q[:3], q[3:], 3)


@pytest.mark.parametrize("edit", [None, "primes"], ids=["other-primes", "no-primes"])
def test_cache_of_other_parameters(tmp_path, edit):
    path = str(tmp_path / "tune.json")
    first = context(54)
    first.autotune(4, cache=path)
    first.close()
    entry = json.load(open(path))
    entry["table"] = [0] * len(entry["table"])       # a table that no tuning gives
    if edit:
        del entry["key"][edit]
    json.dump(entry, open(path, "w"))
    g = context(54 if edit else 61)
    g.autotune(4, cache=path)
    assert any(g.tune_table()) and json.load(open(path))["key"]["primes"] == g.q + g.p
    g.close()


def test_cache_of_the_same_parameters(tmp_path):
    path = str(tmp_path / "tune.json")
    g = context(54)
    g.autotune(4, cache=path)
    entry = json.load(open(path))
    entry["table"] = [0] * len(entry["table"])
    json.dump(entry, open(path, "w"))
    g.autotune(4, cache=path)
    assert not any(g.tune_table())
    g.close()
