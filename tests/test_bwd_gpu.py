"""Parity of bigbird_attn_bwd (tensor-core and CUDA-core gradient kernels) with the fp64 oracle's gradients, through the C-ABI.

Tolerances (max-abs): 1e-4 for fp32 tensors (fp32 arithmetic, sums over up to a few hundred rows); 3e-2 for bf16 tensors
(the gradients are rounded to bf16 on output; |dq|, |dk|, |dv| reach a few units)."""
import numpy as np
import pytest
import torch

import paper_2007_14062_b200 as bb
from paper_2007_14062_b200 import synth
from oracle import bigbird_oracle as O

pytestmark = pytest.mark.gpu
TOL = {"fp32": 1e-4, "bf16": 3e-2}


def _case(dtype, B, H, nb, lengths="full", mode=0, g=2, r=3, w=3, seed=7, b=64, D=64):
    return synth.Workload(f"bwd_{dtype}_{nb}", dtype, B, H, nb * b, D, b, w, g, r, mode, seed=seed, lengths=lengths)


CASES = [
    synth.WORKLOADS["c1_tiny_itc_fp32"],
    _case("fp32", 2, 2, 10, lengths="ragged:64:640"),
    _case("fp32", 1, 2, 7, mode=1, g=1, r=2),
    _case("fp32", 1, 2, 9, b=16, D=32, w=5),                    # another block size and head dimension
    _case("bf16", 2, 2, 12, lengths="ragged:100:768"),
    _case("bf16", 1, 2, 9, mode=1, r=0),
    _case("fp32", 1, 2, 8, b=84, mode=1, g=3, r=0),             # the paper's ETC block size (App. E tables)
    _case("fp32", 1, 2, 6, D=128),                              # the largest head dimension of the CUDA-core kernels
]


@pytest.mark.parametrize("wl", CASES, ids=lambda w: f"{w.name}_{w.lengths}_{w.mode}_{w.b}")
def test_gradients_match_the_oracle(wl, forward=bb.bigbird_attn_fwd_simt):
    dev = torch.device("cuda:0")
    q, k, v = synth.make_qkv(wl)
    gen = torch.Generator().manual_seed(wl.seed + 100)
    dout = torch.randn(q.shape, generator=gen, dtype=torch.float32).to(q.dtype)
    kpm = synth.key_padding_mask(wl)
    if kpm is not None and wl.B > 1:
        kpm[1, 197:] = 0            # a length that is not a multiple of the block size
        kpm[1, :197] = 1
    L = bb.bigbird_build_layout(wl.N, wl.b, wl.w, wl.g, wl.r, wl.seed, wl.H, wl.mode)
    qd, kd, vd, dod = (t.to(dev) for t in (q, k, v, dout))
    md = None if kpm is None else kpm.to(dev)
    out = torch.empty_like(qd)
    lse = torch.empty(q.shape[:3], device=dev, dtype=torch.float32)
    forward(qd, kd, vd, L, md, out, lse, wl.scale)
    dq, dk, dv = (torch.full_like(qd, float("nan")) for _ in range(3))
    bb.bigbird_attn_bwd(qd, kd, vd, out, lse, dod, L, md, dq, dk, dv, wl.scale)
    torch.cuda.synchronize()
    assert bb.bigbird_last_launch_count() == 2
    got = [t.float().cpu().numpy() for t in (dq, dk, dv)]
    assert all(np.isfinite(g).all() for g in got)
    gr = O.Graph(wl.N, wl.b, wl.w, wl.g, wl.r, wl.seed, wl.H, wl.mode)
    want = O.attention_bwd(q.float().numpy(), k.float().numpy(), v.float().numpy(), dout.float().numpy(), gr,
                           None if kpm is None else kpm.numpy(), wl.scale)
    worst = 0.0
    for (bi, h), grads in want.items():
        for g_, w_ in zip(got, grads):
            worst = max(worst, float(np.abs(g_[bi, h] - w_).max()))
    assert worst <= TOL[wl.dtype], (wl.name, worst)
    if kpm is not None:                                         # padded rows: exactly zero
        pad = kpm.numpy() == 0
        for g_ in got:
            assert (g_.transpose(0, 2, 1, 3)[pad] == 0).all()
    L.close()


def test_bad_arguments_are_refused_without_a_launch():
    L = bb.bigbird_build_layout(512, 64, 3, 2, 3, 0, 2, 0)
    t = torch.empty(16, device="cuda:0", dtype=torch.float32)
    ptr = t.data_ptr()
    args = lambda **kw: [kw.get("q", ptr), ptr, ptr, ptr, kw.get("lse", ptr), ptr, L.handle, None, ptr, ptr, ptr, 1, 2, kw.get("N", 512),
                         kw.get("D", 64), 64, 0.125, 0, None]
    # (every call below fails its argument checks before anything is enqueued; a well-formed call is what the parity
    # test above makes)
    assert bb.lib().bigbird_attn_bwd(*args(q=None)) == -1
    assert bb.lib().bigbird_attn_bwd(*args(lse=None)) == -1
    assert bb.lib().bigbird_attn_bwd(*args(N=1024)) == -1       # layout built for another N
    assert bb.lib().bigbird_attn_bwd(*args(D=48)) == -2
    L.close()


# The tensor-core gradient kernels (bf16, b = D = 64) where their schedule can go wrong.  Tolerances as above.
EDGES = [
    _case("bf16", 1, 1, 1, g=1, r=0),                           # one block, one tile without a lower half
    _case("bf16", 1, 1, 4, g=4, r=0),                           # every block global: no sparse tile
    _case("bf16", 1, 2, 7, g=0, r=1),                           # no global block, an unpaired tile
    _case("bf16", 1, 1, 40, g=3, r=2),                          # few heads: tiles of global blocks cut into parts, one of them half empty
    _case("bf16", 1, 1, 120, w=101, lengths="fixed:7000"),      # lists longer than one posted segment
    _case("bf16", 6, 2, 40, lengths="ragged:1:700"),            # mostly padding: many tiles and parts without any step
]


@pytest.mark.parametrize("wl", EDGES, ids=lambda w: f"{w.name}_{w.lengths}_{w.B}_{w.g}{w.r}{w.w}")
def test_tensor_core_gradients_at_the_edges_of_the_schedule(wl):
    test_gradients_match_the_oracle(wl)


@pytest.mark.parametrize("wl", [w for w in CASES if w.dtype == "bf16"] + EDGES, ids=lambda w: f"{w.name}_{w.lengths}_{w.B}_{w.g}{w.r}{w.w}")
def test_tensor_core_forward_and_backward_in_a_row(wl):
    """What a training step does: the gradients of the tensor-core forward pass, queued behind it.  (Its out and lse are as close to
    the oracle's as those of the CUDA-core pass above, so the same tolerance holds.)"""
    test_gradients_match_the_oracle(wl, bb.bigbird_attn_fwd)


@pytest.mark.parametrize("wl", [_case("bf16", 1, 2, 24), _case("bf16", 1, 1, 40, g=3, r=2), _case("bf16", 1, 2, 14, mode=1, r=0)],
                         ids=lambda w: f"{w.name}_{w.mode}")
def test_tensor_core_gradients_keep_sixteen_bits_of_p_and_ds(wl):
    """Against the header's formulas in fp64 from the same bf16 inputs, out and lse.  P and dS enter the products as two bf16
    numbers, 2^-17 of the value off at most, so that nearly all results round to the same bf16 number as the formulas': the formulas
    themselves with P and dS cut to two numbers miss it for 0.25 % of them, 1.2e-4 of the norm, and the kernel 1.3e-4.  Four times
    that is allowed; with one number each it is 42 % and 2.6e-3."""
    dev = torch.device("cuda:0")
    q, k, v = (t.to(dev) for t in synth.make_qkv(wl))
    dout = torch.randn(q.shape, generator=torch.Generator(dev).manual_seed(5), device=dev).to(torch.bfloat16)
    L = bb.bigbird_build_layout(wl.N, wl.b, wl.w, wl.g, wl.r, wl.seed, wl.H, wl.mode)
    out, grads = torch.empty_like(q), [torch.empty_like(q) for _ in range(3)]
    lse = torch.empty(q.shape[:3], device=dev, dtype=torch.float32)
    bb.bigbird_attn_fwd(q, k, v, L, None, out, lse, wl.scale)
    bb.bigbird_attn_bwd(q, k, v, out, lse, dout, L, None, *grads, wl.scale)
    gr = O.Graph(wl.N, wl.b, wl.w, wl.g, wl.r, wl.seed, wl.H, wl.mode)
    A = torch.from_numpy(np.stack([O.build_mask(gr, h) for h in range(wl.H)])).to(dev)
    q, k, v, out, dout, lse = (t.double() for t in (q, k, v, out, dout, lse))
    P = torch.exp(wl.scale * q @ k.mT - lse[..., None]) * A
    dS = P * (dout @ v.mT - (dout * out).sum(-1, keepdim=True))
    for got, want in zip(grads, (wl.scale * dS @ k, wl.scale * dS.mT @ q, P.mT @ dout)):
        rounded = want.to(torch.bfloat16).double()
        off = ((got.double() - rounded).norm() / want.norm()).item()
        assert off <= 5e-4
        assert ((got.double() - want).norm() / want.norm()).item() <= 2e-3     # bf16's rounding itself is 1.7e-3
    L.close()


# Tile shapes of the CUDA-core gradient kernels: see the forward kernel's in test_parity_gpu.py.  Tolerances as above.
SHAPES = [_case("fp32", B, 2, nb, b=b, D=D, g=g, r=2, lengths=f"ragged:{nb * b // 2}:{nb * b}")
          for b, nb, B, D, g in [(1, 12, 1, 32, 1), (5, 12, 1, 64, 1), (16, 12, 1, 128, 1), (33, 12, 1, 64, 1), (96, 12, 1, 64, 1), (97, 12, 1, 32, 1),
                                 (130, 12, 1, 64, 1), (16, 100, 4, 32, 2), (24, 60, 4, 64, 2), (84, 9, 20, 32, 3)]]


@pytest.mark.parametrize("wl", SHAPES, ids=lambda w: f"{w.b}_{w.N // w.b}_{w.B}_{w.D}")
def test_tile_shapes_of_the_cuda_core_gradients(wl):
    test_gradients_match_the_oracle(wl)


# What stands in padded rows must leave no trace, however large (finite: a padded row of k, v, q or dout takes part in tensor-core
# products with probability zero).  Tensor-core gradients, tiles of global blocks whole and cut; the last case pads the tail of a
# global key block.  1e3: scores of a padded key row exceed the row's lse by far more than exp can hold.  3e38: the products
# themselves overflow fp32.
PADDED = [(_case("bf16", 2, 2, 12), 197, 0), (_case("bf16", 1, 1, 40, g=3, r=2), 2001, 0), (_case("bf16", 2, 2, 9, mode=1, g=2, r=0), 500, 100),
          (_case("bf16", 1, 1, 40, mode=1, g=3, r=2), 2560, 130)]


@pytest.mark.parametrize("what,size", [(what, size) for what in ("q", "k", "v", "dout") for size in (1e3, 3e38)])
@pytest.mark.parametrize("wl,valid,gtok", PADDED, ids=lambda x: getattr(x, "name", x))
def test_padded_rows_of_any_finite_size_leave_no_trace(wl, valid, gtok, what, size):
    dev = torch.device("cuda:0")
    kpm = torch.zeros(wl.B, wl.N, dtype=torch.uint8)
    kpm[:, :valid] = 1
    if gtok:
        kpm[:, gtok:wl.g * wl.b] = 0
    pad = (kpm == 0)[:, None, :, None].to(dev)
    t = dict(zip("qkv", (x.to(dev).masked_fill(pad, 0) for x in synth.make_qkv(wl))))
    t["dout"] = torch.randn(t["q"].shape, generator=torch.Generator(dev).manual_seed(3), device=dev).to(torch.bfloat16).masked_fill(pad, 0)
    L = bb.bigbird_build_layout(wl.N, wl.b, wl.w, wl.g, wl.r, wl.seed, wl.H, wl.mode)
    out = torch.empty_like(t["q"])
    lse = torch.empty(out.shape[:3], device=dev, dtype=torch.float32)
    bb.bigbird_attn_fwd(t["q"], t["k"], t["v"], L, kpm.to(dev), out, lse, wl.scale)
    res = []
    for dirty in (False, True):
        if dirty:
            sign = 1 - 2 * (torch.arange(wl.N * wl.D, device=dev).reshape(wl.N, wl.D) % 3 % 2)        # both signs in every row
            t[what] = torch.where(pad, (sign * size).to(torch.bfloat16), t[what])
        grads = [torch.full_like(out, float("nan")) for _ in range(3)]
        bb.bigbird_attn_bwd(t["q"], t["k"], t["v"], out, lse, t["dout"], L, kpm.to(dev), *grads, wl.scale)
        res.append(grads)
    assert bb.bigbird_last_status() == (0, 0)
    for clean, dirty in zip(*res):
        assert torch.equal(clean, dirty)
        assert (dirty.masked_select(pad) == 0).all()
    L.close()
