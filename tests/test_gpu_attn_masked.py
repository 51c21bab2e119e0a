"""Block-causal and block-local attention (dlm_attn_masked) on the GPU against
the oracle's mask variants, with the tolerances of the unmasked attention
tests: bf16 max abs error 2e-2 and the output-scaled bounds, fp32 1e-5;
rows i >= n_b exactly zero. The full mode through the same entry point must
equal dlm_bidir_attn bit for bit."""
import math

import numpy as np
import pytest
import torch

import oracle
from gpu_util import ATTN_TOL_BF16, ATTN_TOL_F32, dev, host_qkv_seq
from paper_2608_02625_gb300 import workloads
from test_gpu_attn import compare, rand_qkv

pytestmark = pytest.mark.gpu

FULL, CAUSAL, LOCAL = 0, 1, 2


def gpu_masked(q, k, v, seq_lens, prompt_lens, mode, block):
    from paper_2608_02625_gb300 import binding as Bn
    d = q.device
    out = torch.full(q.shape, float("nan"), dtype=q.dtype, device=d)
    sl = torch.tensor(np.asarray(seq_lens, dtype=np.int32), device=d)
    pl = torch.tensor(np.asarray(prompt_lens, dtype=np.int32), device=d) if prompt_lens is not None else None
    Bn.dlm_attn_masked(q, k, v, sl, pl, mode, block, out)
    torch.cuda.synchronize()
    assert Bn.device_error(clear=True) == 0
    return out


def run(B, L, Hq, Hkv, D, sl, pl, mode, block, sigma, dtype, seed):
    q, k, v = rand_qkv(B, L, Hq, Hkv, D, sigma, dtype, seed)
    ref = oracle.bidir_attn(q.float().numpy(), k.float().numpy(), v.float().numpy(), sl, mask_mode=mode,
                            block=block, prompt_lens=pl if pl is not None else [0] * B)
    out = gpu_masked(q.to(dev()), k.to(dev()), v.to(dev()), sl, pl, mode, block)
    where = f"mode {mode} block {block} B{B} L{L} {Hq}/{Hkv} D{D} sl {sl} pl {pl}"
    if dtype == "f32":
        return compare(out, ref, sl, ATTN_TOL_F32, where=where)
    return compare(out, ref, sl, ATTN_TOL_BF16, where=where + f" sigma {sigma:.3g}")


@pytest.mark.parametrize("mode", [CAUSAL, LOCAL])
@pytest.mark.parametrize("block", [64, 32, 100, 128, 1000])
@pytest.mark.parametrize("B,L,Hq,Hkv,D,sl,pl", [
    (2, 512, 8, 2, 128, [512, 300], [128, 37]),       # GQA pairs share rows; prompt cut mid sub-tile
    (2, 300, 2, 2, 128, [300, 129], [0, 64]),         # MHA: a unit's two tiles are different row blocks
    (3, 256, 4, 2, 64, [256, 1, 200], [256, 0, 200]),  # all-prompt sequences, n = 1, D = 64
    (1, 640, 4, 1, 128, [640], [256]),                 # c5-shaped lengths
])
def test_bf16_vs_oracle(B, L, Hq, Hkv, D, sl, pl, mode, block):
    run(B, L, Hq, Hkv, D, sl, pl, mode, block, 1 / math.sqrt(D), "bf16", seed=B * L + block + mode)


@pytest.mark.parametrize("mode,block", [(CAUSAL, 64), (LOCAL, 64), (CAUSAL, 7), (LOCAL, 33)])
def test_bf16_peaked(mode, block):
    run(2, 384, 4, 2, 128, [384, 250], [64, 100], mode, block, 1.0, "bf16", seed=block)


@pytest.mark.parametrize("mode,block", [(CAUSAL, 64), (LOCAL, 64), (CAUSAL, 5), (LOCAL, 48)])
def test_f32_vs_oracle(mode, block):
    run(2, 200, 4, 2, 64, [200, 77], [40, 0], mode, block, 1.0, "f32", seed=7 + block)


def test_no_prompt_lens_means_zero():
    run(1, 256, 2, 1, 128, [256], None, LOCAL, 64, 1 / math.sqrt(128), "bf16", seed=5)


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_full_mode_equals_bidir(dtype):
    from paper_2608_02625_gb300 import binding as Bn
    q, k, v = (t.to(dev()) for t in rand_qkv(2, 300, 4, 2, 128, 1.0, dtype, 9))
    sl = [300, 170]
    a = gpu_masked(q, k, v, sl, [50, 20], 0, 64)
    b = torch.empty_like(a)
    Bn.dlm_bidir_attn(q, k, v, torch.tensor(sl, dtype=torch.int32, device=dev()), b)
    torch.cuda.synchronize()
    assert torch.equal(a, b)


def test_prompt_clamp_sets_error_word():
    from paper_2608_02625_gb300 import binding as Bn
    q, k, v = (t.to(dev()) for t in rand_qkv(1, 128, 2, 1, 128, 0.1, "bf16", 2))
    out = torch.empty_like(q)
    Bn.dlm_attn_masked(q, k, v, torch.tensor([100], dtype=torch.int32, device=dev()),
                       torch.tensor([500], dtype=torch.int32, device=dev()), CAUSAL, 64, out)
    torch.cuda.synchronize()
    assert Bn.device_error(clear=True) & 0x1
    ref = oracle.bidir_attn(q.float().cpu().numpy(), k.float().cpu().numpy(), v.float().cpu().numpy(), [100],
                            mask_mode=CAUSAL, block=64, prompt_lens=[500])
    compare(out, ref, [100], ATTN_TOL_BF16, where="clamped prompt")


@pytest.mark.parametrize("mode", [CAUSAL, LOCAL])
def test_full_size_sampled(mode):
    """c3 at full size with 64-token blocks (the drafting block size); the
    oracle recomputes sampled (sequence, head) pairs from host-regenerated q, k, v."""
    from paper_2608_02625_gb300 import synth, synth_gpu
    w = workloads.get("c3_batch32_512")
    d = dev()
    q, k, v = synth_gpu.qkv(w, 0, d)
    sl, pl = w.seq_lens(), w.prompt_lens()
    out = gpu_masked(q, k, v, sl, pl, mode, 64).float().cpu().numpy()
    for b, h in ((0, 0), (7, 13), (31, 31)):
        qs = host_qkv_seq(w, 0, synth.S_Q, b, w.Hq)[:, h:h + 1]
        g = (h * w.Hkv) // w.Hq
        ks = host_qkv_seq(w, 0, synth.S_K, b, w.Hkv)[:, g:g + 1]
        vs = host_qkv_seq(w, 0, synth.S_V, b, w.Hkv)[:, g:g + 1]
        ref = oracle.bidir_attn(qs[None], ks[None], vs[None], [sl[b]], mask_mode=mode, block=64, prompt_lens=[pl[b]])
        err = np.abs(out[b, :, h] - ref[0, :, 0])
        assert err.max() <= ATTN_TOL_BF16, f"mode {mode} b {b} h {h}: {err.max()}"


@pytest.mark.parametrize("mode", [CAUSAL, LOCAL])
def test_workload_full_size(mode):
    """The 32 x 512 workload with its prompt lengths under both block masks (64-token
    blocks, the bench's setting): the whole batch in one launch, the oracle on
    sampled (sequence, query head) pairs from host-generated inputs."""
    from paper_2608_02625_gb300 import synth, synth_gpu
    w = workloads.get("c3_batch32_512")
    q, k, v = synth_gpu.qkv(w, 0, dev())
    n, pl = w.seq_lens(), w.prompt_lens()
    out = gpu_masked(q, k, v, n, pl, mode, 64)
    g_out = out.float()
    for b, heads in ((0, (0, 31)), (9, (5,)), (22, (13, 26)), (31, (7,))):
        hq = host_qkv_seq(w, 0, synth.S_Q, b, w.Hq)
        hk = host_qkv_seq(w, 0, synth.S_K, b, w.Hkv)
        hv = host_qkv_seq(w, 0, synth.S_V, b, w.Hkv)
        for h in heads:
            g = (h * w.Hkv) // w.Hq
            ref = oracle.bidir_attn(hq[None, :, h:h + 1], hk[None, :, g:g + 1], hv[None, :, g:g + 1], [n[b]],
                                    mask_mode=mode, block=64, prompt_lens=[pl[b]])
            compare(g_out[b:b + 1, :, h:h + 1], ref, [n[b]], ATTN_TOL_BF16, where=f"c3 mode {mode} b={b} h={h}")



@pytest.mark.parametrize("mode", [CAUSAL, LOCAL])
@pytest.mark.parametrize("Hq", [2, 40, 80, 152])
def test_f32_values_outside_a_mask_never_reach_a_row(mode, Hq):
    """A NaN or an infinity in v at a key reaches the rows that attend to the key
    and no other, with each query tile of the fp32 kernel (32, 64,
    112, 128 rows)."""
    L, p, block, key = 128, 20, 40, 97   # blocks [20, 60), [60, 100), [100, 128)
    q, k, v = rand_qkv(1, L, Hq, 1, 64, 1.0, "f32", seed=Hq)
    bad = v.clone()
    bad[0, key, 0, ::2] = float("nan")
    bad[0, key, 0, 1::2] = float("inf")
    good, got = (gpu_masked(q.to(dev()), k.to(dev()), x.to(dev()), [L], [p], mode, block) for x in (v, bad))
    attends = torch.zeros(L, dtype=torch.bool, device=dev())
    attends[60:100] = True               # the key's own block
    if mode == CAUSAL:
        attends[100:] = True
    assert torch.equal(got[0, ~attends], good[0, ~attends])
    assert not torch.isfinite(got[0, attends]).any()


@pytest.mark.parametrize("mode", [CAUSAL, LOCAL])
@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_block_of_any_size(dtype, mode):
    """A block of 2^31 - 1 positions: the response is one block."""
    run(2, 300, 4, 2, 64, [300, 200], [70, 0], mode, 2 ** 31 - 1, 0.125, dtype, seed=mode)


@pytest.mark.parametrize("mode", [CAUSAL, LOCAL])
@pytest.mark.parametrize("Hq", [2, 40, 80, 152])
def test_f32_values_of_a_block_never_reach_the_prompt(mode, Hq):
    """The same for a key in a 64-key tile that lies wholly inside the block, of
    which row tiles that begin in the prompt have rows as well."""
    L, p, block, key = 200, 20, 128, 97   # blocks [20, 148), [148, 200); the tile [64, 128)
    q, k, v = rand_qkv(1, L, Hq, 1, 64, 1.0, "f32", seed=Hq + 1)
    bad = v.clone()
    bad[0, key, 0, ::2] = float("nan")
    bad[0, key, 0, 1::2] = float("inf")
    good, got = (gpu_masked(q.to(dev()), k.to(dev()), x.to(dev()), [L], [p], mode, block) for x in (v, bad))
    attends = torch.zeros(L, dtype=torch.bool, device=dev())
    attends[p:p + block] = True
    if mode == CAUSAL:
        attends[p + block:] = True
    assert torch.equal(got[0, ~attends], good[0, ~attends])
    assert not torch.isfinite(got[0, attends]).any()


@pytest.mark.parametrize("mode", [CAUSAL, LOCAL])
@pytest.mark.parametrize("block", [64, 100, 128, 1000])
@pytest.mark.parametrize("B,L,Hq,Hkv,D", [
    (2, 200, 4, 2, 64), (1, 256, 32, 4, 128), (1, 226, 40, 1, 128), (8, 256, 8, 2, 128), (1, 512, 32, 4, 128)])
def test_f32_blocks_of_whole_key_tiles(B, L, Hq, Hkv, D, block, mode):
    """Blocks that contain whole 64-key tiles, with row tiles of 32, 64, 112 and 128
    rows (in this order; 128 twice) that begin in the prompt or end in a later block."""
    for p in (10, 20, 64, 100):
        sl, pl = [L - 5 * b for b in range(B)], [p + b for b in range(B)]
        run(B, L, Hq, Hkv, D, sl, pl, mode, block, 1.0, "f32", seed=L + block + p + mode)


@pytest.mark.parametrize("mode,block", [(CAUSAL, 64), (LOCAL, 64), (CAUSAL, 9), (LOCAL, 20)])
@pytest.mark.parametrize("B,L,Hq,Hkv,D", [
    (2, 337, 24, 2, 128),    # 112-row tiles from head to head, 128-row ones per head when local
    (3, 225, 28, 4, 64),     # 64-row tiles
    (9, 33, 12, 2, 64),      # 32-row tiles; a single key tile: from head to head in both modes
])
def test_f32_tiles_across_heads(B, L, Hq, Hkv, D, mode, block):
    """Tiles whose rows belong to several heads, ragged lengths and prompts, with
    padding rows written by CTAs without rows and by CTAs that have some."""
    sl = [(L, 65, 17, 64, 0, 1, 16, 33, L - 1)[b % 9] for b in range(B)]
    sl = [min(n, L) for n in sl]
    pl = [(0, n // 3, n)[b % 3] for b, n in enumerate(sl)]
    run(B, L, Hq, Hkv, D, sl, pl, mode, block, 1.0, "f32", seed=L + block + mode)


@pytest.mark.parametrize("B,L,Hq,Hkv,D", [
    (3, 1600, 16, 2, 128),    # units taken by the CTAs that are free (12 row tiles and more)
    (7, 1537, 6, 2, 64),      # the same, an odd number of query heads per key/value head
    (6, 1100, 6, 2, 64), (4, 577, 16, 4, 128),    # the same in few rounds, full attention of 4 row tiles and more
    (18, 650, 12, 4, 128), (30, 513, 8, 8, 64),   # block-causal by row tile: odd group, no group
    (40, 129, 8, 2, 128), (73, 300, 4, 1, 64),    # in the order of the heads
])
@pytest.mark.parametrize("mode", [FULL, CAUSAL, LOCAL])
def test_unit_order_bit_identical(mode, B, L, Hq, Hkv, D):
    """Which CTA computes a unit, and when, changes nothing: each sequence of a
    ragged batch as in a call of its own, where every unit has its own CTA."""
    q, k, v = (t.to(dev()) for t in rand_qkv(B, L, Hq, Hkv, D, 1.0, "bf16", L + mode))
    sl = [(L, 1, 0, L - 1, 128, L // 2, 129)[b % 7] for b in range(B)]
    sl = [min(n, L) for n in sl]
    pl = [(0, n // 3, n)[b % 3] for b, n in enumerate(sl)]
    out = gpu_masked(q, k, v, sl, pl, mode, 64)
    for b in range(0, B, max(1, B // 14)):
        one = gpu_masked(q[b:b + 1], k[b:b + 1], v[b:b + 1], sl[b:b + 1], pl[b:b + 1], mode, 64)
        assert torch.equal(out[b:b + 1], one), f"sequence {b}"
    again = gpu_masked(q, k, v, sl, pl, mode, 64)
    assert torch.equal(out, again)
