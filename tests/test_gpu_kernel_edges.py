"""Edges of the kernels' tilings and of the rules that choose between their variants."""
import numpy as np
import pytest
import torch

import oracle
from paper_2501_12369_gb300 import darb

from gpu_helpers import to_np
from test_gpu_density import CFG, RAW, STATE_OF, _case, _device, _t

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2501_12369_gb300 import build
    build.build()
    oracle.build()


def _off_by_one(t):
    """The same values 4 bytes past a 16-byte boundary."""
    flat = torch.empty(t.numel() + 1, dtype=t.dtype, device=t.device)
    v = flat[1:].view(t.shape)
    v.copy_(t)
    assert v.data_ptr() % 16 == 4
    return v


@pytest.mark.parametrize("n", [1, 511, 512, 513, 2048, 2049, 4100])
@pytest.mark.parametrize("deg", [0, 2, 3])
def test_densify_at_block_edges_with_unaligned_moments(n, deg):
    """Row counts around a scatter CTA's 512 and a counted block's 2048 splats, SH rows that are and are
    not multiples of 16 bytes, and moments off the 16-byte boundary (the parameters must be on it)."""
    raw, act, state, accum, count, radius, normals = _case(n, deg, seed=20 + deg)
    ref_raw, ref_act, ref_state, n_ref = oracle.densify(raw, act, state, accum, count, radius, normals, CFG)
    p, st = _device(raw, act, state, deg)
    po, so = _device(raw, act, state, deg, rows=2 * n)
    for s in (st, so):
        for f, t in vars(s).items():
            setattr(s, f, _off_by_one(t))
    n_out = darb.darb_densify(p, st, _t(accum), _t(count), _t(radius), _t(normals), darb.darb_densify_cfg(**CFG), po, so)
    torch.cuda.synchronize()
    rows, _, children = (int(x) for x in to_np(n_out))
    assert rows == n_ref
    for k in RAW:
        got, exact = to_np(getattr(po, k)), children if k == "means" else rows
        np.testing.assert_array_equal(got[:exact], ref_raw[k][:exact], err_msg=k)
        np.testing.assert_allclose(got[:rows], ref_raw[k], rtol=0, atol=2e-6)
        assert np.isnan(got[rows:]).all(), "rows past the output were written"
        for m in ("m", "v"):
            mom = to_np(getattr(so, f"{m}_{STATE_OF[k]}"))
            np.testing.assert_array_equal(mom[:rows], ref_state[f"{m}_{k}"])
            assert np.isnan(mom[rows:]).all()
