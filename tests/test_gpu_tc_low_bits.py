"""n = 50, l = 11 (20 boundary bits): FP_PREC_FP32 takes the faster of the FFMA and the tensor-core
passes, and with the plans it has that is the more accurate FFMA; FP_PREC_TF32X3 takes the tensor
cores.

Tolerance: measured rms errors of a trace are 1.3e-6 (FFMA) and 1.1e-5 (tensor cores)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_precisions_at_20_bits(fp):
    ens = fp.Ensemble(fp.PARALLEL, 50, 11, 11, seed=5)
    t64 = ens.trace_batch(0, 40, fp.PREC_FP64)[0]
    rms = {}
    for prec in (fp.PREC_FP32_RAW, fp.PREC_TF32X3):
        rms[prec] = np.sqrt(np.mean(np.abs(ens.trace_batch(0, 40, prec)[0] - t64) ** 2))
    assert ens.brick_variant(11, fp.PREC_TF32X3)[3] == 4
    assert rms[fp.PREC_FP32_RAW] <= 4e-6 and rms[fp.PREC_TF32X3] <= 4e-5, rms
    ens.close()
