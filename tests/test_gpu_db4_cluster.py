"""The Daubechies-4 prox in one cluster of CTAs, slabs of rows each, against the
FP64 oracle: one CTA to sixteen, slabs of unequal height, transforms down to one
row and one column, images too large for the cluster's shared memory, in place
and not.  An orthonormal pass of four-tap sums is off by at most 4 roundings of
2^-24 in norm, the prox has 4 passes a level, and the threshold is
non-expansive: 16 levels 2^-24 <= 4e-6."""
import numpy as np
import pytest

import synth
from oracle import pp_oracle as O

pytestmark = pytest.mark.gpu

SHAPES = [((2, 2), 1), ((16, 16), 4), ((8, 40), 3), ((24, 64), 3), ((40, 96), 3), ((6, 2), 1), ((112, 16), 4),
          ((176, 104), 3), ((208, 130), 1), ((496, 48), 4), ((384, 384), 3), ((512, 512), 2)]


@pytest.mark.parametrize("shape,levels", SHAPES, ids=["%dx%d_L%d" % (s[0], s[1], l) for s, l in SHAPES])
@pytest.mark.parametrize("inplace", [False, True])
def test_db4_prox_slabs(shape, levels, inplace):
    import torch
    import paper_2204_10252_gb300 as pp
    v = synth.crandn(shape, 7)
    ref = O.prox_l1_db4(v.astype(np.complex128), 0.6, levels)
    xin = torch.from_numpy(v.astype(np.complex64)).cuda()
    out = xin if inplace else torch.empty_like(xin)
    pp.pp_prox_l1_db4(shape, levels, 0.6, xin, out)
    got = out.cpu().numpy().astype(np.complex128)
    assert np.linalg.norm(got - ref) <= 16 * levels * 2.0 ** -24 * np.linalg.norm(v)
