"""The FP64 rate of fea_peak_probe is a peak: within a tenth of two FMA lanes per SM and clock, above what the FP64 tiles
reach (90 % of the unit)."""
import subprocess

import pytest

from tests.helpers import engine

pytestmark = pytest.mark.gpu


def test_fp64_probe_reaches_the_unit():
    import torch
    fea = engine()
    mhz = float(subprocess.check_output(["nvidia-smi", "--query-gpu=clocks.max.sm", "--format=csv,noheader,nounits",
                                         "-i", str(torch.cuda.current_device())], text=True).split()[0])
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert fea.fea_peak_probe(0, 20000) >= 0.9 * (4.0 * sms * mhz * 1e6)
