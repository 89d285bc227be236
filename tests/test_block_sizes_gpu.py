"""The CUDA-core kernels over block sizes at the edges of their tile shapes, against dense attention in fp64."""
import math

import numpy as np
import pytest
import torch

import paper_2007_14062_b200 as bb

pytestmark = pytest.mark.gpu


# Rows per thread: four for 5 (a tile of one warp) and 64; six for 42, 65, 70, 71, 85, 96, 130 and 140; seven for 83 and 84 (a tile of twelve
# rows of threads, with a row to spare and full), 160, 167 and 168 (two such tiles).
@pytest.mark.parametrize("b", [5, 42, 64, 65, 70, 71, 83, 84, 85, 96, 130, 140, 160, 167, 168])
@pytest.mark.parametrize("D", [32, 64])
def test_fp32_forward_and_gradients(b, D):
    B, H, nb = 2, 12, 24
    N = nb * b
    gen = torch.Generator(device="cuda").manual_seed(b)
    q, k, v, dout = (torch.randn((B, H, N, D), generator=gen, device="cuda") for _ in range(4))
    mask = torch.ones((B, N), dtype=torch.uint8)
    mask[1, N - b - 3:] = 0
    mask = mask.cuda()
    L = bb.bigbird_build_layout(N, b, 3, 2, 2, 9, H)
    row_ptr, col_idx = L.export()
    scale = 1.0 / math.sqrt(D)
    out, lse = torch.empty_like(q), torch.empty((B, H, N), device="cuda")
    bb.bigbird_attn_fwd(q, k, v, L, mask, out, lse, scale)
    grads = [torch.empty_like(q) for _ in range(3)]
    bb.bigbird_attn_bwd(q, k, v, out, lse, dout, L, mask, *grads, scale)
    for h in (0, H - 1):
        pairs = np.zeros((nb, nb), dtype=bool)
        for j in range(nb):
            pairs[j, col_idx[row_ptr[h * nb + j]:row_ptr[h * nb + j + 1]]] = True
        attend = torch.from_numpy(pairs).cuda().repeat_interleave(b, 0).repeat_interleave(b, 1)
        for n in range(B):
            keys = mask[n].bool()
            x = [t[n, h].double().requires_grad_() for t in (q, k, v)]
            s = (x[0] @ x[1].T * scale).masked_fill(~(attend & keys[None]), -math.inf)
            want = torch.softmax(s, dim=1) @ x[2]
            (want[keys] * dout[n, h].double()[keys]).sum().backward()
            # fp32 sums of up to 4032 terms: the bounds of the parity and gradient tests
            assert (out[n, h].double()[keys] - want[keys]).abs().max() <= 1e-5
            for g, t in zip(grads, x):
                assert (g[n, h].double() - t.grad).abs().max() <= 1e-4
    L.close()
