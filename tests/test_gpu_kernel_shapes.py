"""Kernels whose tiles, chunks or algorithm depend on the grid, at the sizes where a
tile, a run or a chunk ends: GPU results against the FP64 oracle."""

import numpy as np
import pytest

import oracle
from test_gpu_parity import rel, setup_case

pytestmark = pytest.mark.gpu


# rows shorter and longer than a double-precision stress tile (8 .. 64 columns), heights
# that leave one row in the last tile, chunks of one plane and chunks with a remainder;
# the smallest grids wrap every stencil round the box
@pytest.mark.parametrize("shape", [(8, 4, 8, True), (8, 8, 8, False), (18, 7, 8, True), (36, 29, 9, True),
                                   (64, 9, 12, False), (72, 54, 16, False), (96, 17, 27, True), (162, 13, 8, True)])
@pytest.mark.parametrize("model,extra", [('oldroyd_b', {}), ('saramito', {'Bi': 0.4}), ('fene_p', {'L2': 60.0})])
def test_double_precision_stress_tiles(evp, shape, model, extra):
    import torch
    sim, st, g, prm = setup_case(evp, shape, model, extra, evp.EVP_FP64)
    out = torch.empty((6,) + sim.shape, dtype=torch.float64, device='cuda')
    evp.evp_stress_rhs(sim.handle, out)
    sim.sync()
    ref = oracle.stress_rhs(st.U, st.V, st.W, st.B, g, prm)
    for c in range(6):
        assert rel(out[c].cpu().numpy(), ref[c]) < 1e-12, (c, rel(out[c].cpu().numpy(), ref[c]))
