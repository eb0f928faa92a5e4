"""A barrier timeout stays known until lbm_ensemble_sync has reported it, over
launches that follow it; once reported, the next launch starts anew."""
import pytest

pytestmark = pytest.mark.gpu

CASES = [dict(nx=20, ny=16, nz=12, face=0, Ra=1e5, Pr=0.1, Ste=1.0, Ma=0.2, s0=3.0, derive=True),
         dict(nx=18, ny=14, nz=22, face=1, Ra=3e4, Pr=0.3, Ste=0.5, Ma=0.15, s0=2.5, derive=True)]


@pytest.mark.parametrize("steps", [1, 3, 130])
def test_timeout_survives_later_launches(steps):
    import torch
    assert torch.cuda.is_available()
    import paper_1604_03478_gb300 as P
    from paper_1604_03478_gb300 import _abi
    P.build.build()
    ens = P.Ensemble(CASES)
    ens.step(2)
    ens.sync()
    ens.set_barrier_timeout(20000)
    ens.inject_barrier_fault(0)
    ens.set_barrier_timeout(1 << 24)
    ens.step(steps)
    for _ in range(2):
        with pytest.raises(P.LbmError) as ei:
            ens.sync()
        assert ei.value.status == _abi.LBM_ETIMEOUT
    ens.step(steps)
    try:
        ens.sync()
    except P.LbmError as e:  # the members' states are not meaningful after a timeout
        assert e.status != _abi.LBM_ETIMEOUT
    ens.close()
