"""The transport where its rules on sizes and tables change sides, against the
oracle: allocation with 1, 4 and 16 cells per thread (sides around n^3 = 2^17
and 2^21), and packets settled at home by their quantile word alone, for tables
whose sign change lies at an end, between nodes or on a node."""
import numpy as np
import pytest

import oracle as O
from gpu_helpers import field_dtype, make_fields, new_box, oracle_fields, quantiles, set_state

pytestmark = pytest.mark.gpu


def _compare(cosmo, box, n, Np, q, emis, T):
    set_state(box, np.full(n ** 3, 0.5), T, tally=np.zeros(n ** 3, np.uint32), emis=emis)
    box.transport(3, 1100.0)
    gpu, st = box.tally_np().copy(), box.stats()
    _, _, v4 = oracle_fields(box)
    tally, cnt, _ = O.transport(cosmo, n, 1100.0, 7, 3, Np, box.host("emis"), v4, box.host("T"), q,
                                precision="f32" if box.precision == "mixed" else "f64")
    assert st["crossings"] == cnt["crossings"] and st["absorbed"] == cnt["absorbed"] == Np
    assert np.array_equal(gpu, tally)


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("n", [50, 51, 128, 129])
def test_allocation_rule_edges(cosmo, precision, n):
    Np = 70_001
    rng = np.random.default_rng(n)
    box = new_box(n, precision, n_packets=Np)
    emis = rng.lognormal(0.0, 1.5, n ** 3) * (rng.random(n ** 3) < 0.7)
    emis[-1] = 3.0  # the last block of a ragged side holds weight
    _compare(cosmo, box, n, Np, quantiles(box), emis, rng.uniform(2500.0, 3500.0, n ** 3))
    box.close()


TABLES = {
    "all red": [-3.0, -1.0, -0.5],
    "all blue": [0.5, 1.0, 3.0],
    "two entries": [-1.0, 1.0],
    "two entries, red": [-1.0, -1.0],
    "zeros": [0.0, 0.0],
    "up to zero": [-2.0, -1.0, 0.0],
    "from zero": [0.0, 1.0, 2.0],
    "zero inside": [-2.0, 0.0, 0.0, 0.0, 2.0],
    "tiny end": [-2.0, -1e-12, 2.0],
    "odd count": list(np.linspace(-2.0, 1.5, 4096)),
}


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("table", sorted(TABLES))
def test_home_by_the_quantile_word(cosmo, precision, table):
    from paper_2312_11448_gb300 import rec
    n, Np = 12, 40_003
    rng = np.random.default_rng(len(table))
    d, U = make_fields(n, 0.8, 1.0, 1)
    box = rec.Box(n, d, U, Np, precision=precision, seed=7, quantiles=np.array(TABLES[table]))
    T = rng.uniform(2500.0, 3500.0, n ** 3)
    T[::7] = 0.0  # no thermal width there
    _compare(cosmo, box, n, Np, np.array(TABLES[table], field_dtype(box)), rng.lognormal(0.0, 1.0, n ** 3), T)
    box.close()
