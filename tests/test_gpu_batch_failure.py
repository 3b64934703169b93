"""A batched step's bounded wait that runs out is reported: one wait of an
instance is made on a barrier that nothing arrives at, and returns after its
2 s."""
import ctypes

import pytest

from paper_2506_13072_gb300 import workloads as W

from gpu_common import fvlb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [0, 1, 2, 3])
def test_expired_wait_is_reported(prec):
    F = fvlb()
    expire = F.lib.fvlb_batch_expire_wait
    expire.argtypes, expire.restype = [ctypes.c_void_p, ctypes.c_int], ctypes.c_int
    probs = [W.four_roll(n=n, Wi=0.5, beta=0.5) for n in (12, 33)]
    good, bad = F.Batch(probs, precision=prec), F.Batch(probs, precision=prec)
    for b in (good, bad):
        b.step(3)
        b.synchronize()
    assert expire(bad.h, len(probs)) == F.FVLB_EINVAL
    assert expire(bad.h, 1) == F.FVLB_OK
    for call in (bad.synchronize, lambda: bad.fields(0, F.FVLB_FIELD_U)):
        with pytest.raises(F.FvlbError) as ei:
            call()
        assert ei.value.code == F.FVLB_ETIMEOUT
    good.step(2)
    good.synchronize()          # another batch is not concerned
    good.fields(1, F.FVLB_FIELD_A)
    good.close()
    bad.close()
