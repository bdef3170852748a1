"""complex128 range-Doppler passes: every radix, odd lengths, one batch and several."""
import numpy as np
import pytest
import torch

import oracle
import paper_2208_10939_gb300 as pkg

pytestmark = pytest.mark.gpu


# a column a block and fewer columns than multiprocessors; equal runs in one
# batch; two blocks a multiprocessor with several batches (the last, shorter)
@pytest.mark.parametrize("O,N,M", [(1, 2, 32), (2, 3, 36), (1, 9, 54), (3, 16, 48), (2, 128, 384),
                                   (5, 18, 972), (1, 1024, 192), (7, 81, 1024)])
def test_rdm_fp64(O, N, M):
    rng = np.random.default_rng(O * 1009 + N * 13 + M)
    cube = rng.normal(size=(O, N, M)) + 1j * rng.normal(size=(O, N, M))
    ref = oracle.range_doppler_map(cube)
    out = torch.empty((M, N), dtype=torch.float32, device="cuda")
    pkg.bart_form_rdm_static(torch.from_numpy(cube).cuda(), out, O, N, M)
    got = out.cpu().numpy().astype(np.float64)
    # one float32 rounding of a cell, and FP64 transforms of at most 20 radix-2
    # levels: 20 x 2^-53 x the largest amplitude's share, well below 1e-13 of it
    assert np.all(np.abs(got - ref) <= 2.0 ** -24 * ref + 1e-13 * ref.max())
