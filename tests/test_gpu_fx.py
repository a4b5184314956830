"""FP64 paths in fixed-point arithmetic (mcg_fx.cuh) against the FP64 oracle
at the edges of their ranges: lattices of extent 2 (a neighbour reached from
both sides), ragged tails of the blocks, several fields per call, staple
weights up to the limit of the fixed-point step and just above it (the FP64
kernels)."""
import numpy as np
import pytest

import oracle
from paper_0807_0264_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _pack(mcg, Us, dims):
    return mcg.mcg_pack_links(torch.from_numpy(np.ascontiguousarray(np.stack(Us))).cuda(), dims)


# rho (6 |cp| + 18 |cr|) at, below and above the limit 1; n even and odd (the
# two buffers); the oracle rounds ~150 times per link and step at 1.1e-16
# relative to entries of at most 1: 2e-14 per step
@pytest.mark.parametrize("rho,eps,n", [(1 / 6, 1.0, 3), (0.1667, 1.0, 2), (0.07751937984496124, -0.25, 2),
                                       (-0.1, 1.0, 1), (0.06, -0.25, 5), (1e-9, 1.0, 2), (0.0, 0.5, 1)])
@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (6, 2, 10, 4), (4, 14, 2, 6)])
def test_fixed_point_smear(dims, rho, eps, n):
    from paper_0807_0264_gb300 import mcg

    Us = [synth.make_field(dims, w, s) for w, s in ((0.5, 1), (3.0, 2), (0.0, 3))]
    S = mcg.mcg_unpack_links(mcg.mcg_smear(_pack(mcg, Us, dims), dims, rho, eps, n), dims).cpu().numpy()
    for U, s in zip(Us, S):
        assert np.abs(s - oracle.smear(dims, U, rho, eps, n)).max() < 2e-14 * n
