"""Lattices whose fused measurement cannot be driven phase by phase are refused there
with the calls that take them named; those calls work."""
import numpy as np
import pytest

from workloads import FP32_COMPRESSED, FP64_PLAIN, HOT

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,frozen", [(FP64_PLAIN, False), (FP64_PLAIN, True), (FP32_COMPRESSED, True)])
def test_refusal(precision, frozen):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    import paper_1310_7087_gb300 as q
    lat = q.Lattice(3, 4, 4, 5.7, 1, precision, HOT, 7, field_mode=q.QCD_FIELD_FROZEN if frozen else q.QCD_FIELD_LINKS)
    for call in (lambda: lat.phase(q.QCD_OVERRELAX_MEASURE, 1, 2, 5), lambda: q.qcd_measure_fused_finish(lat.h)):
        with pytest.raises(q.QcdError, match="phase by phase .*qcd_working_sweep") as e:
            call()
        assert e.value.code == q.QCD_ERR_NOT_SUPPORTED
    got = np.array(q.qcd_working_sweep(lat.h, 1, 1, 5))
    p, l = lat.measure()
    assert np.abs(got - np.array(p + l)).max() < 1e-6
    lat.close()
