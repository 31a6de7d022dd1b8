"""Bounded waits of the single-box launches: every form of the persistent
substep (and the adjoint's evaluations) gives up at a zero limit, rec_sync
reports it once, also when the state has been set anew in between, and the
context then steps to the result of one that never timed out."""
import numpy as np
import pytest

from gpu_helpers import make_fields

pytestmark = pytest.mark.gpu

FORMS = [("fp64", "tally"), ("fp64", "full"), ("fp64", "partial"), ("mixed", "tally"), ("mixed", "full"),
         ("mixed", "partial")]


def _box(precision, mixing, n=32):
    from paper_2312_11448_gb300 import rec
    d, U = make_fields(n, 0.8, 1.0, seed=3)
    kw = dict(f_alpha=0.6) if mixing == "partial" else {}
    return rec.Box(n, d, U, 200_000, precision=precision, mixing=mixing, seed=7, **kw)


def _run(box, U, z0=1300.0, z1=1295.0):
    box.tally.zero_()
    box.vel4.copy_(U)
    box.state_init(z0)
    box.transport(0, z0)
    box.step(0, z0, z1)


def _fields(box):
    return [box.host(k).copy() for k in ("x", "T", "vel4", "emis")]


def _expires(box):
    from paper_2312_11448_gb300 import rec
    with pytest.raises(rec.RecError) as ei:
        box.sync()
    assert ei.value.status == rec.REC_ETIMEOUT
    box.sync()  # reported once


@pytest.mark.parametrize("sync_first", [True, False])
@pytest.mark.parametrize("precision,mixing", FORMS)
def test_substep_expiry_and_recovery(precision, mixing, sync_first):
    ref = _box(precision, mixing)
    U = ref.vel4.clone()
    _run(ref, U)
    ref.sync()
    want = _fields(ref)
    ref.close()
    box = _box(precision, mixing)
    box.set_wait_limit(0)
    _run(box, U)
    if sync_first:
        _expires(box)
    box.set_wait_limit(1 << 22)
    _run(box, U)  # sets the state anew: it steps, whether the expiry has been reported or not
    if not sync_first:
        _expires(box)
    assert box.stats()["flags"] & 8 == 0
    for a, b in zip(_fields(box), want):
        np.testing.assert_array_equal(a, b)
    box.close()


def test_refresh_keeps_an_expiry_for_the_report():
    box = _box("fp64", "tally")
    U = box.vel4.clone()
    box.set_wait_limit(0)
    _run(box, U)
    box.refresh(1295.0)
    _expires(box)
    box.close()


def test_batch_refresh_keeps_an_expiry_for_the_report():
    from paper_2312_11448_gb300 import rec
    boxes = [(n, *make_fields(n, 0.8, 1.0, seed=n), 40_000) for n in (16, 24)]
    b = rec.Batch(boxes, precision="mixed", mixing="tally", seed=9)
    b.set_wait_limit(0)
    b.state_init(1400.0)
    b.transport(0, 1400.0)
    b.step(0, 1400.0, 1395.0)
    b.refresh(1395.0)
    _expires(b)
    b.close()


@pytest.mark.parametrize("mixing", ["tally", "full"])
def test_adjoint_expiry_and_recovery(mixing):
    import torch
    box = _box("fp64", mixing)
    z0, z1, n3 = 1300.0, 1295.0, box.n3
    box.state_init(z0)
    x, T = box.x.clone(), box.T.clone()
    g = torch.Generator(device="cuda")
    g.manual_seed(1)
    tally = torch.randint(0, 20, (n3,), generator=g, device="cuda", dtype=torch.int32)
    xb, Tb = (torch.randn(n3, generator=g, device="cuda", dtype=torch.float64) for _ in range(2))

    def reverse():
        out = [xb.clone(), Tb.clone(), torch.zeros_like(xb), torch.zeros_like(xb)]
        box.step_adjoint(0, z0, z1, x, T, None, tally, out[0], out[1], None, out[2], out[3], Xe_bar_out=0.7)
        return out

    want = reverse()
    box.sync()
    box.set_wait_limit(0)
    reverse()
    _expires(box)
    box.set_wait_limit(1 << 22)
    got = reverse()
    box.sync()
    for a, b in zip(got, want):
        assert torch.equal(a, b)
    box.close()
