"""The SU(3) FP32 phases whose staples are shared by six warps, at the sizes where
they change: a ragged last CTA, more than one wave of CTAs (programmatic
launches), the last size that splits and the first that does not.  Every kernel of
a sweep against the oracle from the state the one before left (the FP32 bar of
test_gpu_parity), and the working sweep's sums against the separate measurement."""
import numpy as np
import pytest

import test_gpu_parity as parity
from workloads import FP32_COMPRESSED, HOT

pytestmark = pytest.mark.gpu
q = parity.q


@pytest.mark.parametrize("Ns,Nt,flux", [(10, 2, 1), (20, 4, 0), (20, 6, 2), (16, 14, 1)])
def test_phases(q, Ns, Nt, flux):
    parity.run_kernel_by_kernel(q, (3, FP32_COMPRESSED, Ns, Nt, 5.7, flux))


@pytest.mark.parametrize("Ns,Nt,flux8", [(10, 2, 0), (20, 6, 1), (16, 14, 0)])
def test_working_sweep(q, Ns, Nt, flux8):
    a = q.Lattice(3, Ns, Nt, 5.7, 1, FP32_COMPRESSED, HOT, 7, flux8=flux8)
    got = np.array(q.qcd_working_sweep(a.h, 2, 2, 5))
    p, l = a.measure()
    assert np.abs(got - np.array(p + l)).max() < 1e-6
    a.close()
