"""Contexts without the optional scratch (the compact velocity copy, the FP64
cell cache) against ones with it: the same tallies and counters, the same bits
of a step, the adjoint to rounding."""
import numpy as np
import pytest

from gpu_helpers import make_fields

pytestmark = pytest.mark.gpu


def _make(monkeypatch, level, make):
    monkeypatch.setenv("REC_SCRATCH", level)
    out = make()
    monkeypatch.delenv("REC_SCRATCH")
    return out


def _velocities(U, n):
    U = U.copy()
    U[n ** 3 // 3] *= 1e4  # one cell beyond the copy's scale
    return U


@pytest.mark.parametrize("level", ["least", "copy"])
@pytest.mark.parametrize("precision,n,halo", [("mixed", 31, 0), ("mixed", 64, 8), ("fp64", 32, 0), ("fp64", 33, 0), ("fp64", 64, 8)])
def test_single_box(monkeypatch, level, precision, n, halo):
    from paper_2312_11448_gb300 import rec
    d, U = make_fields(n, 0.8, 1.0, seed=3)
    got = []
    for lv in ("", level):
        box = _make(monkeypatch, lv, lambda: rec.Box(n, d, _velocities(U, n), 100_003, precision=precision, mixing="tally", seed=7))
        if halo:
            box.set_tuning(march_halo=halo, tile=16, march_blocks_per_sm=2)
        box.state_init(1250.0)
        box.transport(2, 1250.0)
        tally, st = box.tally_np().copy(), box.stats()
        box.step(2, 1250.0, 1245.0)
        box.sync()
        got.append([tally, np.array([st[k] for k in ("emitted", "absorbed", "capped", "crossings", "queued")])] +
                   [box.host(k) for k in ("x", "T", "vel4", "emis")])
        box.close()
    for a, b in zip(*got):
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
def test_batch(monkeypatch, precision):
    from paper_2312_11448_gb300 import rec
    sizes = [13, 16, 24]
    fields = [make_fields(n, 0.8, 1.0, n) for n in sizes]
    got = []
    for lv in ("", "least"):
        b = _make(monkeypatch, lv, lambda: rec.Batch([(n, d, _velocities(U, n), 20_003) for n, (d, U) in zip(sizes, fields)],
                                                     precision=precision, mixing="tally", seed=7))
        b.state_init(1250.0)
        b.transport(2, 1250.0)
        got.append([b.tally_np(i).copy() for i in range(3)] + [np.array([s["crossings"] for s in b.stats()])])
        b.close()
    for x, y in zip(*got):
        np.testing.assert_array_equal(x, y)


@pytest.mark.parametrize("level", ["least", "copy"])
@pytest.mark.parametrize("mixing", ["tally", "full", "partial"])
def test_fp64_step_without_the_cell_cache(monkeypatch, level, mixing):
    from paper_2312_11448_gb300 import rec
    n = 33
    d, U = make_fields(n, 0.8, 1.0, seed=3)
    kw = dict(f_alpha=0.6) if mixing == "partial" else {}
    got = []
    for lv in ("", level):
        box = _make(monkeypatch, lv, lambda: rec.Box(n, d, U, 50_000, precision="fp64", mixing=mixing, seed=7, n_sub=2, **kw))
        box.state_init(1250.0)
        box.transport(2, 1250.0)
        box.step(2, 1250.0, 1245.0)
        box.sync()
        got.append([box.host(k) for k in ("x", "T", "vel4", "emis")])
        box.close()
    for a, b in zip(*got):
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("mixing", ["tally", "full"])
def test_adjoint_without_the_cell_cache(monkeypatch, mixing):
    """The two forms of the reverse sweep round differently: a few units of 1.1e-16 of the largest value."""
    import torch
    from paper_2312_11448_gb300 import rec
    n = 21
    d, U = make_fields(n, 0.8, 1.0, seed=3)
    got = []
    for lv in ("", "least"):
        box = _make(monkeypatch, lv, lambda: rec.Box(n, d, U, 1000, precision="fp64", mixing=mixing, seed=7))
        box.state_init(1250.0)
        g = torch.Generator(device="cuda")
        g.manual_seed(2)
        tally = torch.randint(0, 40, (box.n3,), generator=g, device="cuda", dtype=torch.int32)
        out = [torch.randn(box.n3, generator=g, device="cuda", dtype=torch.float64) for _ in range(2)]
        out += [torch.zeros_like(out[0]), torch.zeros_like(out[0])]
        box.step_adjoint(0, 1250.0, 1240.0, box.x.clone(), box.T.clone(), None, tally, out[0], out[1], None, out[2],
                         out[3], Xe_bar_out=0.7)
        box.sync()
        got.append([t.cpu().numpy() for t in out])
        box.close()
    for a, b in zip(*got):
        assert np.abs(a - b).max() <= 1e-12 * np.abs(a).max()
