"""LBM_FLAG_TEST_WAIT_TIMEOUT on any instance of a small 16-bit batch: its waits
run out, on whichever instance the flag is, and lbm_batch_sync reports it."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2308_16597_gb300 import lbm, workloads as W  # noqa: E402


@pytest.mark.parametrize("flagged", [0, 1, 2])
def test_timeout_is_reported_whichever_instance_waits(flagged):
    prm = W.base_params(0.05, 0.71, 1e-4)
    sims = [lbm.Simulation(W.cavity(300, 40), None, prm, storage=lbm.LBM_STORE_BF16,
                           flags=lbm.LBM_FLAG_TEST_WAIT_TIMEOUT if k == flagged else 0) for k in range(3)]
    b = lbm.Batch(sims)
    b.step(1)
    with pytest.raises(lbm.LbmError) as e:
        b.sync()
    assert e.value.code == lbm.LBM_ETIMEOUT
    b.close()
    for s in sims:
        s.close()
