"""GPU: the tiles the library chooses by itself, at the sizes where they can go
wrong: the tensor-core collision filter (reg = 0), the row tiles of the FP32
distance map (reg = 0), Life runs of more than 16 steps, the fused cost-model
kernels and the scaled FP16 planes of the tensor-core distance map."""
import numpy as np
import pytest

from gpu_util import dev, rel_err, tri
from paper_1609_01490_gb300 import inputs

pytestmark = pytest.mark.gpu


# ------------------------------------------------------------ FP32 distances --
@pytest.mark.parametrize("prec", ["BF16X6", "BF16X3"])
def test_tc_edm_row_scales(orc, prec):
    # rows from 2^-40 to 2^40, zero rows, rows whose largest feature dwarfs the
    # others: every distance within the 1e-5 the split is built for
    import torch
    t, D = tri(), dev()
    n, d = 400, 96
    x = inputs.edm_normal_points(n, d, seed=5)
    rng = np.random.default_rng(7)
    x = (x * np.exp2(rng.integers(-40, 41, size=(n, 1)))).astype(np.float32)
    x[::37] = 0.0
    x[3::29, 0] *= np.float32(2.0 ** 20)
    out = torch.empty(n * (n + 1) // 2, device=D)
    p = getattr(t, prec)
    ws = torch.empty(t.tri_edm_workspace_size(n, d, p), dtype=torch.uint8, device=D)
    t.tri_edm(torch.from_numpy(x).to(D), out, prec=p, workspace=ws)
    assert rel_err(out.cpu().numpy(), orc.edm_packed(x)) <= 1e-5
