"""A substep as a launch per pass, which is what runs where a persistent
cooperative launch cannot, against the persistent one: the same sums in the
same order, so the same bits, in every form and in the adjoint."""
import numpy as np
import pytest

import oracle as O
from gpu_helpers import make_fields, oracle_fields, set_state

pytestmark = pytest.mark.gpu


def _box(monkeypatch, sel, precision, mixing, n):
    from paper_2312_11448_gb300 import rec
    monkeypatch.setenv("REC_NEWTON", sel)
    d, U = make_fields(n, 0.8, 1.0, seed=3)
    kw = dict(f_alpha=0.6) if mixing == "partial" else {}
    return rec.Box(n, d, U, 1000, precision=precision, mixing=mixing, seed=7, n_sub=2 if mixing != "tally" else 1, **kw)


def _state(cosmo, box, z):
    rng = np.random.default_rng(11)
    d, _, _ = oracle_fields(box)
    return (O.saha_xe(cosmo, z, d) * 0.98, O.background(cosmo, z)["Tg"] * (1.0 + 0.01 * rng.standard_normal(d.size)),
            rng.poisson(20 * d ** 1.5).astype(np.uint32))


@pytest.mark.parametrize("mixing", ["tally", "full", "partial"])
@pytest.mark.parametrize("precision,n", [("fp64", 5), ("fp64", 33), ("mixed", 33), ("mixed", 72)])
def test_launch_per_pass_equals_the_persistent_substep(cosmo, monkeypatch, precision, mixing, n):
    out = []
    for sel in ("plain", "passes"):
        box = _box(monkeypatch, sel, precision, mixing, n)
        x, T, tally = _state(cosmo, box, 1250.0)
        set_state(box, x, T, tally=tally)
        box.refresh(1250.0)
        box.timing(True)
        box.step(0, 1250.0, 1240.0)
        box.sync()
        st = box.stats()
        assert st["flags"] == 0
        out.append([box.host(k) for k in ("x", "T", "vel4", "emis")] + [np.array([st["lam"], st["X_e"], st["newton_passes"]])])
        out.append(box.kernel_times()["rec_step"][1])
        box.close()
    for a, b in zip(out[0], out[2]):
        np.testing.assert_array_equal(a, b)
    assert out[3] == out[1] + 11 * (2 if mixing != "tally" else 1)


@pytest.mark.parametrize("mixing", ["tally", "full"])
def test_adjoint_with_a_launch_per_pass(cosmo, monkeypatch, mixing):
    import torch
    out = []
    for sel in ("plain", "passes"):
        monkeypatch.setenv("REC_NEWTON", sel)
        from paper_2312_11448_gb300 import rec
        d, U = make_fields(21, 0.8, 1.0, seed=3)
        box = rec.Box(21, d, U, 1000, precision="fp64", mixing=mixing, seed=7)
        x, T, tally = (torch.as_tensor(v if v.dtype != np.uint32 else v.view(np.int32)).cuda()
                       for v in _state(cosmo, box, 1250.0))
        g = torch.Generator(device="cuda")
        g.manual_seed(2)
        b = [torch.randn(box.n3, generator=g, device="cuda", dtype=torch.float64) for _ in range(2)]
        b += [torch.zeros_like(x), torch.zeros_like(x)]
        box.step_adjoint(0, 1250.0, 1240.0, x, T, None, tally, b[0], b[1], None, b[2], b[3], Xe_bar_out=0.7)
        box.sync()
        out.append([t.cpu().numpy() for t in b])
        box.close()
    for a, b in zip(*out):
        np.testing.assert_array_equal(a, b)
