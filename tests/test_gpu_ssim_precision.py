"""Precision of the image loss where the variances cancel: nearly equal, flat images."""
import numpy as np
import pytest
import torch

import oracle
from paper_2501_12369_gb300 import darb

from gpu_helpers import to_np

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2501_12369_gb300 import build
    build.build()
    oracle.build()


@pytest.mark.parametrize("a,b", [(0.8, 0.79), (0.51, 0.5), (0.93, 0.95), (0.3, 0.31), (0.77, 0.77), (1.0, 0.99)])
def test_ssim_of_flat_images(a, b):
    """Inside a flat image A2 and B2 are C2 = 9e-4 but for rounding, some 2^-24 a b each.  Only their quotient matters,
    and they share that rounding: they differ by the variance of x - y, whose 22 additions round to 22 U
    (a - b)^2, below 3e-7 of C2.  A1 and B1 differ by (m_x - m_y)^2, off by 88 U a |a - b| <= 1e-7, and six
    products round to 6 U: together below 1e-6."""
    x, y = (np.full((3, 48, 64), v, np.float32) for v in (a, b))
    ref_loss, _, ref_ssim = oracle.l1_dssim_loss(x, y, 0.2)
    _, loss = darb.darb_l1_dssim_loss(torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda(), 0.2)
    assert abs(to_np(loss)[1] - ref_ssim) <= 1e-6
    assert abs(to_np(loss)[0] - ref_loss) <= 1e-6
