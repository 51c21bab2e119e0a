"""Step A2 (vocabulary reduction) on the GPU against the oracle.

argmax is bit-exact (exact compare, lowest index wins); conf and lse are within
the relative tolerances of gpu_util."""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import check_vocab, dev, host_logit_rows
from paper_2608_02625_gb300 import synth, workloads

pytestmark = pytest.mark.gpu


def gpu_vocab(x: torch.Tensor):
    from paper_2608_02625_gb300 import binding as Bn
    N = x.shape[0] if x.dim() == 2 else x.shape[0] * x.shape[1]
    am = torch.full((N,), -1, dtype=torch.int32, device=x.device)
    cf = torch.full((N,), -1.0, dtype=torch.float32, device=x.device)
    ls = torch.full((N,), -1.0, dtype=torch.float32, device=x.device)
    Bn.dlm_vocab_confidence(x, am, cf, ls)
    torch.cuda.synchronize()
    return am.cpu().numpy(), cf.cpu().numpy(), ls.cpu().numpy()


def to_dev(x_f32: np.ndarray, dtype: str) -> torch.Tensor:
    t = torch.from_numpy(np.ascontiguousarray(x_f32, dtype=np.float32))
    return (t.to(torch.bfloat16) if dtype == "bf16" else t).to(dev())


@pytest.mark.parametrize("name", ["c1_tiny_f32", "c2_single_512"])
def test_workload_all_rows(name):
    w = workloads.get(name)
    from paper_2608_02625_gb300 import synth_gpu
    x = synth_gpu.logits(w, 0, dev())
    am, cf, ls = gpu_vocab(x)
    rows = np.arange(w.N)
    ref = oracle.vocab_confidence(host_logit_rows(w, 0, rows))
    check_vocab(am, cf, ls, *ref, where=name)


@pytest.mark.parametrize("name", ["c3_batch32_512", "c4_long_2048", "c5_heavy_4step"])
def test_workload_sampled_rows(name):
    """Full-size launch; the oracle recomputes ~180 rows one by one (random,
    and at the edges of waves of CTAs and of sequences)."""
    w = workloads.get(name)
    from paper_2608_02625_gb300 import synth_gpu
    tok, msk = w.initial_state()
    t_tok = torch.from_numpy(tok.reshape(-1)).to(dev())
    t_msk = torch.from_numpy(msk.reshape(-1)).to(dev())
    x = synth_gpu.logits(w, 0, dev(), t_tok, t_msk)
    am, cf, ls = gpu_vocab(x)
    rng = np.random.default_rng(5)
    # 160 random rows, plus rows at the edges of waves of resident CTAs (4 per
    # SM on 152 SMs) and of sequences.
    wave = 4 * 152
    edges = [r for k in range(1, 4) for r in (k * wave - 1, k * wave) if r < w.N]
    seq_edges = [r for b in (0, 1, w.B // 2, w.B - 1) for r in (b * w.L, b * w.L + w.L - 1)]
    rows = np.unique(np.concatenate([[0, w.N - 1], edges, seq_edges, rng.integers(0, w.N, 160)]))
    ref = oracle.vocab_confidence(host_logit_rows(w, 0, rows, tok.reshape(-1)[rows], msk.reshape(-1)[rows]))
    check_vocab(am[rows], cf[rows], ls[rows], *ref, where=name)
    del x
    torch.cuda.empty_cache()


def planted(N, V, seed, sigma=3.0):
    rng = np.random.default_rng(seed)
    return (rng.standard_normal((N, V)) * sigma).astype(np.float32)


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("N,V", [(1, 1), (3, 7), (2, 8), (5, 1001), (64, 4096), (1, 151552), (7, 151553),
                                 (300, 32000)])
def test_shapes(dtype, N, V):
    x = planted(N, V, N * 7 + V)
    t = to_dev(x, dtype)
    ref = oracle.vocab_confidence(t.float().cpu().numpy())
    check_vocab(*gpu_vocab(t), *ref, where=f"{dtype} {N}x{V}")


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_ties_and_neg_inf(dtype):
    N, V = 6, 151552
    x = planted(N, V, 3)
    x[0, [5, 77777, 150000]] = 40.0          # ties in different threads / cluster chunks
    x[1, :] = -np.inf
    x[1, [123456, 99]] = [2.0, 2.0]          # only two finite entries, tied
    x[2, ::3] = -np.inf
    x[3, :] = 1.5                            # all equal
    x[4, V - 1] = 50.0                       # maximum at the last index
    x[5, 0] = 50.0
    t = to_dev(x, dtype)
    am, cf, ls = gpu_vocab(t)
    ref = oracle.vocab_confidence(t.float().cpu().numpy())
    check_vocab(am, cf, ls, *ref, where="ties")
    assert am[0] == 5 and am[1] == 99 and am[3] == 0 and am[4] == V - 1 and am[5] == 0


def test_strided_rows_and_3d():
    N, V = 40, 5000
    wide = to_dev(planted(N, V + 24, 11), "bf16")
    x = wide[:, 8:8 + V]                     # rows 16-byte aligned, row stride V + 24
    ref = oracle.vocab_confidence(x.float().cpu().numpy())
    check_vocab(*gpu_vocab(x), *ref, where="strided")
    x3 = to_dev(planted(4 * 10, V, 12), "bf16").reshape(4, 10, V)
    ref3 = oracle.vocab_confidence(x3.reshape(40, V).float().cpu().numpy())
    check_vocab(*gpu_vocab(x3), *ref3, where="3d")
    odd = wide[:, 3:3 + V]                   # rows not 16-byte aligned
    ref_odd = oracle.vocab_confidence(odd.float().cpu().numpy())
    check_vocab(*gpu_vocab(odd), *ref_odd, where="unaligned")


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("N,V,pad", [(1000, 1003, 5), (2000, 64, 0), (700, 40000, 8), (900, 12, 4)])
def test_many_rows_ragged(dtype, N, V, pad):
    """More rows than one wave of resident CTAs (the staged scan), with row
    lengths that leave a scalar tail, tiny rows (most threads idle) and padded
    row strides."""
    x = planted(N, V + pad, N + V)
    t = to_dev(x, dtype)[:, :V]
    ref = oracle.vocab_confidence(t.float().cpu().numpy())
    check_vocab(*gpu_vocab(t), *ref, where=f"{dtype} {N}x{V}+{pad}")


@pytest.mark.parametrize("dtype,N,V", [("bf16", 200, 151552), ("f32", 160, 65536), ("bf16", 100, 151552)])
def test_split_rows_several_per_cluster(dtype, N, V):
    """Few long rows (at most two per SM): each row is split over a cluster, and
    with these counts a cluster takes several rows in turn (alternating partial
    slots); ties planted across the chunk boundaries of a cluster."""
    x = planted(N, V, N + V + 1)
    chunk = V // 8
    for r in range(0, N, 7):
        x[r, [chunk - 1, 3 * chunk + 5, V - 1]] = 30.0   # equal maxima in different CTAs' chunks
    t = to_dev(x, dtype)
    am, cf, ls = gpu_vocab(t)
    ref = oracle.vocab_confidence(t.float().cpu().numpy())
    check_vocab(am, cf, ls, *ref, where=f"{dtype} {N}x{V}")
    assert all(am[r] == chunk - 1 for r in range(0, N, 7))


def test_c4_zipf_full_size_planted_ties():
    """The long-draft workload at full size (16384 rows of the Zipf(1.1) prior
    plus N(0, 1)), with equal maxima planted in sampled rows at positions that
    fall to different threads, warps and staging slots of the row kernel, and
    to different CTAs' chunks of the split-row clusters (a 256-row slice); the
    lowest index must win everywhere."""
    from paper_2608_02625_gb300 import synth_gpu
    w = workloads.get("c4_long_2048")
    x = synth_gpu.logits(w, 0, dev())
    V = w.V
    rng = np.random.default_rng(44)
    rows = np.unique(np.concatenate([[0, 1, 255, w.N - 1], rng.integers(0, w.N, 24)]))
    pos = np.array([V // 8 - 1, 3 * (V // 8) + 5, V // 2 + 2048 * 8 + 3, V - 1])   # first planted index wins
    peak = float(x[torch.from_numpy(rows).to(dev())].float().max().item()) + 16.0   # exact in bf16 (an integer)
    peak = float(torch.tensor(peak).to(torch.bfloat16).float())
    for r in rows:
        x[int(r), torch.from_numpy(pos).to(dev())] = peak
    am, cf, ls = gpu_vocab(x)
    ref = oracle.vocab_confidence(host_rows_planted(w, rows, pos, peak))
    check_vocab(am[rows], cf[rows], ls[rows], *ref, where="c4 planted ties")
    assert np.all(am[rows] == pos[0])
    sl = rows[rows < 256]
    sub = x[:256]
    ref_s = oracle.vocab_confidence(host_rows_planted(w, sl, pos, peak))
    outs = gpu_vocab(sub)
    check_vocab(outs[0][sl], outs[1][sl], outs[2][sl], *ref_s, where="c4 planted ties, 256 rows, clusters")
    assert np.all(outs[0][sl] == pos[0])
    del x
    torch.cuda.empty_cache()


def host_rows_planted(w, rows, pos, peak):
    x = host_logit_rows(w, 0, rows)
    x[:, pos] = np.float32(peak)
    return x


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("N,V", [(3, 1), (5, 3), (4, 17), (9, 65537), (40, 4099), (700, 5), (700, 33), (1300, 4097),
                                 (650, 9001)])
def test_rows_off_16_byte_boundaries(dtype, N, V):
    """Rows packed under an odd V, seen from every starting element: a cluster,
    a CTA and a warp per row, rows shorter than one vector; equal maxima before,
    inside and after a row's whole vectors, and -inf there."""
    for off in range(8 if dtype == "bf16" else 4):
        x = planted(N, V, N + V + off)
        x[0, [0, V // 2, V - 1]] = 40.0
        x[1, [V - 1, V // 2]] = 40.0
        x[2, :] = -np.inf
        x[2, V - 1 - off % V] = -3.0
        flat = to_dev(np.concatenate([np.full(off, 99.0, np.float32), x.reshape(-1)]), dtype)
        t = flat[off:].view(N, V)
        ref = oracle.vocab_confidence(t.float().cpu().numpy())
        check_vocab(*gpu_vocab(t), *ref, where=f"{dtype} {N}x{V} off {off}")


@pytest.mark.parametrize("dtype,peak", [("bf16", 77.5), ("f32", 77.3), ("f32", -301.7)])
@pytest.mark.parametrize("N,V", [(2, 40001), (300, 9001), (700, 1000)])
def test_large_maxima_cost_no_accuracy(dtype, peak, N, V):
    """m log2(e) rounded is off by up to 2^-18 here (half an ulp of 435), the same
    way for every term; the sum must not keep that. Left are the rounding of
    ex2.approx (2^-22), of x - m from the FMA and of the sums (a few 2^-24)."""
    rng = np.random.default_rng(V)
    x = (peak - rng.integers(0, 9, (N, V)) / 2).astype(np.float32)
    t = to_dev(x, dtype)
    _, conf, lse = gpu_vocab(t)
    y = t.double()
    exact = torch.exp(y.max(1).values - torch.logsumexp(y, 1)).cpu().numpy()
    assert np.abs(conf / exact - 1).max() <= 2.0 ** -20


@pytest.mark.parametrize("dtype,V", [("bf16", 51201), ("bf16", 110001), ("f32", 17001)])
def test_choice_of_clusters(dtype, V):
    """Clusters of 16, 8 and 4, a CTA per row, clusters of 2 and a CTA per row again,
    with every number of rows around which the choice turns on 152 SMs."""
    x = planted(210, V, V)
    x[::7, V - 1] = 40.0
    x[::7, V // 2] = 40.0
    full = to_dev(x, dtype)
    ref = oracle.vocab_confidence(full.float().cpu().numpy())
    for N in (9, 10, 21, 22, 33, 34, 50, 51, 75, 76, 113, 114, 115, 147, 148, 149, 152, 153, 202, 203, 210):
        check_vocab(*gpu_vocab(full[:N]), *(r[:N] for r in ref), where=f"{dtype} {N}x{V}")


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("N,V", [(12, 151553), (700, 1003), (300, 9001), (500, 9001)])
def test_maxima_of_any_size(dtype, N, V):
    """Rows whose maximum, or whose first maxima, lie anywhere between the type's
    ends: suppressed entries at the lowest value, whole vectors of them at the
    start of every thread, rows of nothing else; in a cluster, a warp and a CTA
    (staged, from registers) per row."""
    low, high = (float(f(torch.bfloat16 if dtype == "bf16" else torch.float32)) for f in
                 (lambda t: torch.finfo(t).min, lambda t: torch.finfo(t).max))
    rng = np.random.default_rng(V)
    x = planted(N, V, N + V)
    x[0, :] = low
    x[1, :] = low
    x[1, V - 1] = 2.5
    x[2, :V // 2] = low
    x[3, rng.random(V) < 0.9] = low
    x[4, [V // 3, V // 2]] = high
    x[5, :] = high
    x[6, :] = np.where(rng.random(V) < 0.5, 2.5e38, 3.0e38)
    x[7, :V - 20] = -1e30
    x[8, :V // 2] = -3e10
    x[9, :] = -1e9
    x[10, :] = np.float32(2.0 ** 30) - 64.0 * rng.integers(0, 4, V).astype(np.float32)
    x[11, :] = 300007.0 + rng.integers(-8, 1, V) / 4
    t = to_dev(x, dtype)
    ref = oracle.vocab_confidence(t.float().cpu().numpy())
    check_vocab(*gpu_vocab(t), *ref, where=f"{dtype} {N}x{V}")


@pytest.mark.parametrize("N", [38, 152, 304, 456])
def test_leaves_shared_memory_to_other_streams(N):
    """A reduction that has one to three CTAs on every SM (clusters, a CTA per row)
    leaves a kernel of another stream that needs 50 KB of shared memory room
    beside it: the small call, issued later, ends first."""
    from paper_2608_02625_gb300 import binding as Bn
    d = dev()
    V = 2 ** 31 // N // 8 * 8               # 4.3 GB: most of a millisecond
    x = torch.zeros(N, V, dtype=torch.bfloat16, device=d)
    outs = [torch.empty(N, dtype=t, device=d) for t in (torch.int32, torch.float32, torch.float32)]
    q = torch.zeros(1, 32, 1, 64, device=d)
    k, v, out = torch.zeros_like(q), torch.zeros_like(q), torch.zeros_like(q)
    streams = [torch.cuda.Stream(d) for _ in range(2)]
    for _ in range(3):
        ends = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        torch.cuda.synchronize()
        with torch.cuda.stream(streams[0]):
            Bn.dlm_vocab_confidence(x, *outs)
            ends[0].record()
        with torch.cuda.stream(streams[1]):
            Bn.dlm_bidir_attn(q, k, v, None, out)
            ends[1].record()
        torch.cuda.synchronize()
    assert ends[1].elapsed_time(ends[0]) > 0.1
