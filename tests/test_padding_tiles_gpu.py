"""Tiles without a token, and sequences that end inside, before and at the edges of tiles: what the schedulers of the tensor-core
kernels clear themselves.  Results and gradients start from NaN, so that rows nobody writes are found."""
import math

import numpy as np
import pytest
import torch

import paper_2007_14062_b200 as bb

pytestmark = pytest.mark.gpu

# B, H, nb, g, mode, lengths: few tiles per stream and many; an odd number of sparse blocks; global tiles cut into parts or not, with
# and without tokens; lengths at block and tile edges
CASES = [
    (3, 2, 8, 2, 0, [0, 1, 512]),
    (2, 3, 13, 2, 0, [64, 65]),
    (3, 4, 70, 3, 1, [0, 4480, 128]),
    (2, 2, 96, 2, 0, [4097, 191]),
    (40, 8, 16, 2, 0, None),
]


def _lengths(B, nb, lengths):
    return np.array(lengths) if lengths else np.random.RandomState(7).randint(0, nb * 64 + 1, B)


@pytest.mark.parametrize("case", CASES, ids=lambda c: f"B{c[0]}_H{c[1]}_nb{c[2]}_g{c[3]}_mode{c[4]}")
@pytest.mark.parametrize("entry", ["fwd", "static"])
def test_rows_of_tiles_without_tokens(case, entry):
    B, H, nb, g, mode, lengths = case
    N = nb * 64
    lens = _lengths(B, nb, lengths)
    gen = torch.Generator(device="cuda").manual_seed(3)
    q, k, v, dout = (torch.randn((B, H, N, 64), generator=gen, device="cuda").to(torch.bfloat16) for _ in range(4))
    mask = torch.from_numpy((np.arange(N)[None] < lens[:, None]).astype(np.uint8)).cuda()
    rows = mask.bool()[:, None, :].expand(B, H, N)
    L = bb.bigbird_build_layout(N, 64, 3, g, 3, 5, H, mode)
    scale = 1.0 / math.sqrt(64)

    def empty():
        return torch.full_like(q, float("nan")), torch.full((B, H, N), float("nan"), device="cuda")

    out, lse = empty()
    fwd = bb.bigbird_attn_fwd if entry == "fwd" else bb.bigbird_attn_fwd_static
    fwd(q, k, v, L, mask, out, lse, scale)
    ref, ref_lse = empty()
    bb.bigbird_attn_fwd_simt(q, k, v, L, mask, ref, ref_lse, scale)
    assert (bb.bigbird_last_status() if entry == "fwd" else bb.bigbird_last_status_static())[0] == 0
    assert (out[~rows] == 0).all() and (lse[~rows] == -math.inf).all()
    if rows.any():
        # bf16 probabilities and results against fp32 arithmetic on the same bf16 inputs: the bounds of the parity tests
        assert (out[rows].float() - ref[rows].float()).abs().max() <= 2e-2
        assert (lse[rows] - ref_lse[rows]).abs().max() <= 1e-3
    if entry == "static":
        L.close()
        return
    grads = [empty()[0] for _ in range(3)]
    bb.bigbird_attn_bwd(q, k, v, out, lse, dout, L, mask, *grads, scale)
    assert bb.bigbird_last_status()[0] == 0
    for x in grads:
        assert (x[~rows] == 0).all() and torch.isfinite(x[rows].float()).all()
    # the fp32 gradients of the same inputs
    f = [t.float() for t in (q, k, v, out, dout)]
    want = [torch.full_like(f[0], float("nan")) for _ in range(3)]
    bb.bigbird_attn_bwd(f[0], f[1], f[2], f[3], lse, f[4], L, mask, *want, scale)
    for x, y in zip(grads, want):
        # the gradients are rounded to bf16 once (2^-9 of a value) and carry 16 bits of P and dS (the bound of the gradient tests)
        err = torch.linalg.norm((x[rows].float() - y[rows]).double()) if rows.any() else 0.0
        assert err <= (2.0 ** -8 + 5e-4) * torch.linalg.norm(y[rows].double())
    L.close()


def test_streams_that_end_with_a_tile_of_one_step():
    """Short sequences leave streams whose last tile has a single step: its message to the epilogue and the end mark follow each other
    before the epilogue has taken the tile in front."""
    B, H, nb = 40, 8, 16
    N = nb * 64
    mask = torch.from_numpy((np.arange(N)[None] < _lengths(B, nb, None)[:, None]).astype(np.uint8)).cuda()
    q, k, v = (torch.randn((B, H, N, 64), device="cuda").to(torch.bfloat16) for _ in range(3))
    out, lse = torch.empty_like(q), torch.empty((B, H, N), device="cuda")
    L = bb.bigbird_build_layout(N, 64, 3, 2, 3, 5, H, 0)
    for fwd, status in ((bb.bigbird_attn_fwd, bb.bigbird_last_status), (bb.bigbird_attn_fwd_static, bb.bigbird_last_status_static)):
        for _ in range(100):
            fwd(q, k, v, L, mask, out, lse, 0.125)
            assert status()[0] == 0
    L.close()


@pytest.mark.parametrize("entry", ["fwd", "static"])
def test_parts_without_tokens_leave_nothing_of_their_scratch(entry):
    """Tiles of global blocks that are cut into parts and hold no token: nothing is written for such a part, and the merge must not let
    through what an earlier call left in its place."""
    B, H, nb = 1, 2, 70
    N = nb * 64
    L = bb.bigbird_build_layout(N, 64, 3, 4, 3, 5, H, 1)
    fwd = bb.bigbird_attn_fwd if entry == "fwd" else bb.bigbird_attn_fwd_static
    q, k, v = (torch.randn((B, H, N, 64), device="cuda").to(torch.bfloat16) for _ in range(3))
    mask = torch.ones((B, N), dtype=torch.uint8, device="cuda")
    res = []
    for dirty in (q, torch.full_like(q, float("nan")), q * 1e19):       # what the earlier call computes: sums, NaN, infinities
        out, lse = torch.full_like(q, float("nan")), torch.full((B, H, N), float("nan"), device="cuda")
        mask.fill_(1)
        fwd(dirty, dirty, v, L, mask, out, lse, 0.125)
        mask[:, :128] = 0                                                # the first pair of global blocks
        fwd(q, k, v, L, mask, out, lse, 0.125)
        assert (out[:, :, :128] == 0).all() and (lse[:, :, :128] == -math.inf).all() and torch.isfinite(out.float()).all()
        res.append((out, lse))
    assert all(torch.equal(x, y) for r in res[1:] for x, y in zip(r, res[0]))
    L.close()


@pytest.mark.parametrize("padded", [False, True])
def test_lists_of_many_segments(padded):
    """Lists that are posted in five segments, three tiles per stream: while the scheduler waits for room for one stream's segments the
    other one ends a tile, and its last product is issued only when its next tile has been posted; the epilogue must serve the first
    stream meanwhile."""
    B, H, nb = 1, 4, 420
    N = nb * 64
    q, k, v = (torch.randn((B, H, N, 64), generator=torch.Generator(device="cuda").manual_seed(i), device="cuda").to(torch.bfloat16) for i in range(3))
    mask = (torch.arange(N, device="cuda")[None] < N - 70).to(torch.uint8) if padded else None
    L = bb.bigbird_build_layout(N, 64, 401, 1, 0, 5, H, 0)
    out, lse, ref, ref_lse = torch.empty_like(q), torch.empty((B, H, N), device="cuda"), torch.empty_like(q), torch.empty((B, H, N), device="cuda")
    for _ in range(10):
        bb.bigbird_attn_fwd(q, k, v, L, mask, out, lse, 0.125)
        assert bb.bigbird_last_status()[0] == 0
    bb.bigbird_attn_fwd_simt(q, k, v, L, mask, ref, ref_lse, 0.125)
    rows = slice(0, N - 70 if padded else N)
    # the bounds of the parity tests
    assert (out[:, :, rows].float() - ref[:, :, rows].float()).abs().max() <= 2e-2
    assert (lse[:, :, rows] - ref_lse[:, :, rows]).abs().max() <= 1e-3
    L.close()


@pytest.mark.parametrize("shape", [(9, 1, 1, 0, 0), (33, 3, 0, 5, 0), (24, 5, 3, 0, 1), (120, 101, 2, 3, 0), (16, 3, 2, 40, 0)],
                         ids=lambda s: "nb%d_w%d_g%d_r%d_mode%d" % s)
@pytest.mark.parametrize("padded", [False, True])
def test_gradients_of_steps_that_the_halves_of_a_tile_share(shape, padded):
    """Tiles whose halves have equally many blocks of their own, unequally many or none, and lists longer than a posted segment."""
    nb, w, g, r, mode = shape
    B, H, N = 2, 2, nb * 64
    gen = torch.Generator(device="cuda").manual_seed(nb)
    q, k, v, dout = (torch.randn((B, H, N, 64), generator=gen, device="cuda").to(torch.bfloat16) for _ in range(4))
    lens = np.array([N - 70, max(1, N // 3)])
    mask = torch.from_numpy((np.arange(N)[None] < lens[:, None]).astype(np.uint8)).cuda() if padded else None
    L = bb.bigbird_build_layout(N, 64, w, g, r, 5, H, mode)
    out, lse = torch.empty_like(q), torch.empty((B, H, N), device="cuda")
    bb.bigbird_attn_fwd(q, k, v, L, mask, out, lse, 0.125)
    grads = [torch.full_like(q, float("nan")) for _ in range(3)]
    bb.bigbird_attn_bwd(q, k, v, out, lse, dout, L, mask, *grads, 0.125)
    assert bb.bigbird_last_status()[0] == 0
    f = [t.float() for t in (q, k, v, out, dout)]
    want = [torch.empty_like(f[0]) for _ in range(3)]
    bb.bigbird_attn_bwd(f[0], f[1], f[2], f[3], lse, f[4], L, mask, *want, 0.125)
    for x, y in zip(grads, want):               # the bound of the test above
        assert torch.linalg.norm((x.float() - y).double()) <= (2.0 ** -8 + 5e-4) * torch.linalg.norm(y.double())
    L.close()


# The launch takes the form of the kernel with shared steps where the halves of the layout's tiles have many blocks of their own.  With
# it: short lists; lists of several posted segments; a little more than a fifth of the steps saved.  Without it: an ETC layout with
# about a sixth saved, lists of several segments with hardly any.
@pytest.mark.parametrize("shape,shared", [((70, 1, 2, 0, 0), True), ((200, 3, 2, 60, 0), True), ((16, 3, 2, 3, 0), True), ((66, 3, 2, 0, 1), False),
                                          ((140, 131, 1, 0, 0), False)], ids=lambda s: "nb%d_w%d_g%d_r%d_mode%d" % s if isinstance(s, tuple) else str(s))
@pytest.mark.parametrize("padded", [False, True])
def test_gradients_with_and_without_shared_steps(shape, shared, padded):
    nb, w, g, r, mode = shape
    L = bb.bigbird_build_layout(nb * 64, 64, w, g, r, 5, 2, mode)
    globals_ = set(range(g)) if mode else set(range((g + 1) // 2)) | set(range(nb - g // 2, nb))
    sparse = [j for j in range(nb) if j not in globals_]
    blocks = steps = 0
    for ptr, idx in (L.export(), L.export_transposed()):
        rows = [set(idx[ptr[i]:ptr[i + 1]]) for i in range(2 * nb)]
        for h in range(2):
            for a, b in zip(sparse[::2], sparse[1::2] + [None]):
                upper, lower = rows[h * nb + a], rows[h * nb + b] if b is not None else rows[h * nb + a]
                blocks += len(upper | lower)
                steps += len(upper & lower) + max(len(upper - lower), len(lower - upper))
    assert (5 * (blocks - steps) > blocks) == shared     # (the case is on the side that it stands for)
    L.close()
    test_gradients_of_steps_that_the_halves_of_a_tile_share(shape, padded)
