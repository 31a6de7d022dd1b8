"""The march's bound on the compact velocity copy against the oracle's exact
test: tallies and crossing counts are bit-identical whatever the velocities,
at the edges of the copy's bricks (4 cells), its axis bits and both wraps."""
import numpy as np
import pytest

import oracle as O
from gpu_helpers import new_box, oracle_fields, quantiles, set_state

pytestmark = pytest.mark.gpu


def _velocities(kind, n, rng):
    v = rng.normal(0.0, 2.0, (n ** 3, 3))
    if kind == "still":
        v[:] = 0.0
    elif kind == "tiny":
        v *= 1e-30
    elif kind == "spike":  # the scale is set by one cell: the bound is loose everywhere else
        v[n ** 3 // 2] = (3.0e4, -2.0e4, 1.0e4)
    elif kind == "infinite":  # no scale: every cell takes the exact test
        v[n ** 3 // 2] = (np.inf, 0.0, -np.inf)
    return v


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("kind", ["normal", "still", "tiny", "spike", "infinite"])
@pytest.mark.parametrize("n", [1, 2, 3, 5, 8, 31, 33])
def test_bound_keeps_the_exact_result(cosmo, precision, kind, n):
    Np = 20_011
    rng = np.random.default_rng(100 * n + len(kind))
    box = new_box(n, precision, n_packets=Np)
    v = _velocities(kind, n, rng)
    box.vel4[:, :3].copy_(box.torch.as_tensor(v))
    emis = rng.lognormal(0.0, 1.0, n ** 3)
    if kind == "infinite" and n > 1:
        emis[n ** 3 // 2] = 0.0  # its packets would never come into resonance
    elif kind == "infinite":
        box.close()
        return
    T = rng.uniform(2500.0, 3500.0, n ** 3)
    set_state(box, np.full(n ** 3, 0.5), T, tally=np.zeros(n ** 3, np.uint32), emis=emis)
    box.transport(3, 1100.0)
    gpu, st = box.tally_np().copy(), box.stats()
    _, _, v4 = oracle_fields(box)
    tally, cnt, _ = O.transport(cosmo, n, 1100.0, 7, 3, Np, box.host("emis"), v4, box.host("T"), quantiles(box),
                                precision="f32" if precision == "mixed" else "f64")
    assert st["crossings"] == cnt["crossings"] and st["absorbed"] == cnt["absorbed"] == Np
    assert np.array_equal(gpu, tally)
    box.close()
