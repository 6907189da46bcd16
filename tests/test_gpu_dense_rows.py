"""The FP32 dense layer without allocation above 8 rows: a row has the same bits alone among 9 rows as among any number, at any
place, also where the partials of all rows exceed the scratch and the call takes several launches."""

import numpy as np
import pytest

from gpu_common import require_gpu

pytestmark = pytest.mark.gpu


# (splits of K on 152 multiprocessors, rows to a launch): (50, 128), (152, 64), (8, 2112), (1, 20)
@pytest.mark.parametrize("N,K,most", [(300, 32768, 300), (128, 110592, 300), (24, 4104, 700), (100000, 8, 20)])
def test_rows_do_not_depend_on_their_batch(N, K, most):
    F = require_gpu()
    import torch

    g = torch.Generator(device="cuda").manual_seed(N)
    x = torch.rand((9, K), generator=g, device="cuda") - 0.5
    w = torch.rand((N, K), generator=g, device="cuda") - 0.5
    b = torch.rand((N,), generator=g, device="cuda")

    def run(rows):
        y = torch.full((len(rows), N), float("nan"), device="cuda")
        F.fusion_cnn_dense_noalloc(rows.contiguous(), w, b, len(rows), N, K, False, y,
                                   torch.cuda.current_stream().cuda_stream)
        return y.cpu().numpy()

    nine = run(x)
    splits = max(1, min(128, K // 2048))
    for B in sorted({10, 17, 64, 65, 100, 129, most}):
        if B > most or splits * B * N > F.FUSION_NOALLOC_MAX_PARTIALS:
            continue
        at = [(5 * i) % 9 for i in range(B)]
        np.testing.assert_array_equal(run(x[at]), nine[at])
