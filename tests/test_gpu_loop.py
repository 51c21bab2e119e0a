"""The recorded multi-pass loop (dlm_loop_*): one graph launch repeats a refine
pass on the GPU until no confident edit remains or max_steps passes have run
(Sec. 4.2's T_r passes; Appendix C.4's early stop).

Against the oracle (oracle.refine_passes): the host regenerates each pass's
logits from the state the previous oracle pass left, with the same seeded
generator the GPU pass uses, and runs the oracle's vocabulary reduction and
update. The pass count, tokens, mask and edit counts must be identical; the
decision-margin protocol applies per pass, and these cases have no position
within the confidence tolerance of a decision in any pass (checked here), so
the comparison is exact. Also: the same pass issued pass by pass from the
host, which must agree with the graph launch bit for bit."""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import ambiguous_for, dev
from paper_2608_02625_gb300 import synth, workloads

pytestmark = pytest.mark.gpu


class Case:
    """c5-shaped state (128 x 640 scaled to B sequences); the model stand-in is
    the seeded generator: q, k, v and logits whose peaks follow the current
    tokens, regenerated by every pass from the state the last pass left."""

    def __init__(self, B, edit_threshold=None, V=None, seq_lens=None, static=False):
        from paper_2608_02625_gb300 import binding as Bn
        d = dev()
        base = workloads.get("c5_heavy_4step")
        w = workloads.scaled(base, B=B, V=V or base.V, name=f"c5_b{B}")
        self.static = static
        self.w = w
        tok, msk = w.initial_state()
        self.tok0 = torch.from_numpy(tok).to(d)
        self.msk0 = torch.from_numpy(msk).to(d)
        self.tok = self.tok0.clone()
        self.msk = self.msk0.clone()
        dt = torch.bfloat16
        self.q = torch.empty((w.B, w.L, w.Hq, w.D), dtype=dt, device=d)
        self.k = torch.empty((w.B, w.L, w.Hkv, w.D), dtype=dt, device=d)
        self.v = torch.empty((w.B, w.L, w.Hkv, w.D), dtype=dt, device=d)
        self.out = torch.empty_like(self.q)
        self.logits = torch.empty((w.N, w.V), dtype=dt, device=d)
        self.am = torch.empty((w.B, w.L), dtype=torch.int32, device=d)
        self.cf = torch.empty((w.B, w.L), dtype=torch.float32, device=d)
        self.ls = torch.empty((w.B, w.L), dtype=torch.float32, device=d)
        self.ne = torch.zeros(w.B, dtype=torch.int32, device=d)
        self.ws = torch.zeros(w.B, dtype=torch.int32, device=d)
        self.steps = torch.full((1,), -1, dtype=torch.int32, device=d)
        self.prompt_np = w.prompt_lens()
        self.seqlen_np = w.seq_lens() if seq_lens is None else np.asarray(seq_lens, dtype=np.int32)
        self.prompt = torch.from_numpy(self.prompt_np).to(d)
        self.seqlen = torch.from_numpy(self.seqlen_np).to(d)
        tau = w.edit_threshold[0] if edit_threshold is None else edit_threshold
        self.tau = tau
        self.params = Bn.RefineParams(tau, w.remask_k, w.remask_frac, w.mask_id, self.prompt, self.seqlen)
        seed = w.step_seed(0)
        self.keys = [synth.stream_key(seed, s) for s in (synth.S_Q, synth.S_K, synth.S_V)]
        self.spec = w.logit_spec(0)

    def reset(self):
        self.tok.copy_(self.tok0)
        self.msk.copy_(self.msk0)

    def one_pass(self):
        """Model stand-in, attention, then the fused vocabulary reduction and
        in-place update (tokens / mask are read and rewritten by every pass)."""
        from paper_2608_02625_gb300 import binding as Bn
        from paper_2608_02625_gb300 import synth_gpu
        for t, key in zip((self.q, self.k, self.v), self.keys):
            synth_gpu.fill_normal_(t, key, self.w.qkv_sigma)
        Bn.dlm_bidir_attn(self.q, self.k, self.v, self.seqlen, self.out)
        synth_gpu.fill_logits_(self.logits, self.spec, 0, self.tok.view(-1), self.msk.view(-1))
        if self.static:
            Bn.dlm_refine_step_static(self.logits, self.tok, self.msk, self.params, self.am, self.cf, self.ls,
                                      self.tok, self.msk, self.ne)
        else:
            Bn.dlm_refine_step(self.logits, self.tok, self.msk, self.params, self.am, self.cf, self.ls,
                               self.tok, self.msk, self.ne, self.ws)

    def state(self):
        return self.tok.cpu().numpy(), self.msk.cpu().numpy(), self.ne.cpu().numpy()


def oracle_loop(c: Case, max_steps: int):
    """oracle.refine_passes on host-regenerated logits; also returns the number
    of positions within the confidence tolerance of a decision, over all passes."""
    w = c.w
    amb = [0]

    def logits_for(tok, msk, t):
        x = c.spec.rows_f32(np.arange(w.N), tok.reshape(-1), msk.reshape(-1))
        x = synth.bf16_bits_to_f32(synth.f32_to_bf16_bits(x))
        am, cf, _ = oracle.vocab_confidence(x)
        amb[0] += int(ambiguous_for(c.tau, w.remask_k, w.remask_frac, cf.reshape(w.B, w.L), (tok, msk),
                                    am.reshape(w.B, w.L), np.clip(c.prompt_np, 0, None),
                                    np.clip(c.seqlen_np, 0, w.L)).sum())
        return x

    tok0, msk0 = c.tok0.cpu().numpy(), c.msk0.cpu().numpy()
    r = oracle.refine_passes(tok0, msk0, logits_for, max_passes=max_steps, edit_threshold=c.tau,
                             remask_k=w.remask_k, remask_frac=w.remask_frac, mask_id=w.mask_id,
                             prompt_lens=c.prompt_np, seq_lens=c.seqlen_np)
    return r["passes"], (r["tokens"], r["mask"], r["n_edits"]), amb[0]


def host_loop(c: Case, max_steps: int):
    from paper_2608_02625_gb300 import binding as Bn
    c.reset()
    steps = 0
    for s in range(max_steps):
        c.one_pass()
        torch.cuda.synchronize()
        steps = s + 1
        if not bool((c.ne > 0).any()):
            break
    assert Bn.device_error(clear=True) == 0
    return steps, c.state()


def record(c: Case, max_steps: int, stream):
    from paper_2608_02625_gb300 import binding as Bn
    with torch.cuda.stream(stream):
        Bn.dlm_loop_begin(c.steps)
        try:
            c.one_pass()
        except BaseException:
            Bn.dlm_loop_cancel()
            raise
        return Bn.dlm_loop_end(c.ne, max_steps, c.steps)


def graph_loop(c: Case, loop, stream, allowed_bits=0):
    """One launch of the recorded loop from the initial state; the device error
    word may hold only `allowed_bits` afterwards (it is cleared)."""
    from paper_2608_02625_gb300 import binding as Bn
    with torch.cuda.stream(stream):
        c.reset()
        c.steps.fill_(-1)
        loop.launch()
    torch.cuda.synchronize()
    bits = Bn.device_error(clear=True)
    assert bits & ~allowed_bits == 0, f"device error word {bits:#x}"
    return int(c.steps.item()), c.state()


def same(a, b, where):
    for name, x, y in zip(("tokens", "mask", "n_edits"), a, b):
        assert np.array_equal(x, y), f"{where}: {name} differs at {np.argwhere(x != y)[:8].tolist()}"


def check_against_oracle(c: Case, max_steps: int, expect: str, allowed_bits=0, launches=2):
    ref_steps, ref, amb = oracle_loop(c, max_steps)
    assert amb == 0, f"{amb} positions within the confidence tolerance of a decision: not an exact case"
    if expect == "no_edit":      # stops after the first pass without a confident edit
        assert 2 <= ref_steps < max_steps and not ref[2].any()
    elif expect == "budget":     # edits remain, the budget ends the loop
        assert ref_steps == max_steps and ref[2].any()
    elif expect == "one":        # nothing can be edited: one pass
        assert ref_steps == 1 and not ref[2].any()
    stream = torch.cuda.Stream()
    loop = record(c, max_steps, stream)
    try:
        for launch in range(launches):
            steps, got = graph_loop(c, loop, stream, allowed_bits)
            assert steps == ref_steps, f"launch {launch}: {steps} passes, oracle {ref_steps}"
            same(got, ref, f"launch {launch} against the oracle")
    finally:
        loop.close()


@pytest.mark.parametrize("max_steps,edit_threshold,expect", [(8, None, "no_edit"), (1, None, "budget"),
                                                             (8, 2.0, "one")])
def test_loop_matches_oracle(max_steps, edit_threshold, expect):
    """Two c5-shaped sequences (256 prompt + 384 response, V = 8192): the early
    stop, a budget that ends the loop while edits remain, and a threshold no
    confidence reaches."""
    check_against_oracle(Case(2, edit_threshold, V=8192), max_steps, expect)


def test_clamped_length_does_not_stop_the_loop():
    """A sequence length above L is clamped to L (a defined result, flagged
    with DLM_DEVERR_LENGTH); the loop goes on to its early stop as the oracle,
    which clamps the same way, does."""
    from paper_2608_02625_gb300 import binding as Bn
    L = workloads.get("c5_heavy_4step").L
    Bn.device_error(clear=True)
    c = Case(2, V=8192, seq_lens=[L, L + 7])
    check_against_oracle(c, 8, "no_edit", allowed_bits=0x1, launches=1)
    # The bit was set by the launch (graph_loop cleared it): run once more and look.
    stream = torch.cuda.Stream()
    loop = record(c, 8, stream)
    try:
        with torch.cuda.stream(stream):
            c.reset()
            loop.launch()
        torch.cuda.synchronize()
        assert Bn.device_error(clear=True) == 0x1
    finally:
        loop.close()


def test_timeout_bit_stops_the_loop():
    """A pass whose kernels record DLM_DEVERR_TIMEOUT (here: the bounded-wait
    self-test recorded after the refine step) leaves undefined outputs, so the
    loop stops after it although edits remain."""
    from paper_2608_02625_gb300 import binding as Bn
    c = Case(2, V=8192)
    ref_steps, _, _ = oracle_loop(c, 8)
    assert ref_steps >= 2
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        Bn.dlm_loop_begin(c.steps)
        try:
            c.one_pass()
            Bn.dlm_selftest_wait_timeout(10000)
        except BaseException:
            Bn.dlm_loop_cancel()
            raise
        loop = Bn.dlm_loop_end(c.ne, 8, c.steps)
    try:
        steps, state = graph_loop(c, loop, stream, allowed_bits=0x2)
        assert steps == 1 and state[2].any()
    finally:
        loop.close()


def test_recorded_static_step_matches_oracle():
    """The recorded pass may use dlm_refine_step_static: dlm_loop_begin takes
    the address of the device error word before the capture starts."""
    check_against_oracle(Case(2, V=8192, static=True), 8, "no_edit")


@pytest.mark.parametrize("max_steps,edit_threshold", [(8, None), (1, None), (8, 2.0)])
def test_loop_matches_host_driven_passes(max_steps, edit_threshold):
    c = Case(16, edit_threshold)
    ref_steps, ref = host_loop(c, max_steps)
    if edit_threshold is not None and edit_threshold > 1:
        assert ref_steps == 1            # no confidence reaches the threshold: stop after one pass
    elif max_steps > 1:
        assert 2 <= ref_steps <= max_steps   # the first pass edits, so a second one runs
    stream = torch.cuda.Stream()
    loop = record(c, max_steps, stream)
    try:
        for launch in range(2):   # a loop can be launched again; each launch restarts the count
            steps, got = graph_loop(c, loop, stream)
            assert steps == ref_steps, f"launch {launch}: {steps} passes, host-driven {ref_steps}"
            same(got, ref, f"launch {launch}")
    finally:
        loop.close()


def test_recording_does_not_run_the_pass():
    """Calls made while recording are captured, not executed."""
    from paper_2608_02625_gb300 import binding as Bn
    c = Case(2)
    c.reset()
    c.ne.fill_(-3)
    torch.cuda.synchronize()
    stream = torch.cuda.Stream()
    loop = record(c, 4, stream)
    torch.cuda.synchronize()
    try:
        assert int(c.ne[0].item()) == -3 and torch.equal(c.tok, c.tok0)
        steps, _ = graph_loop(c, loop, stream)
        assert 1 <= steps <= 4
    finally:
        loop.close()
    assert Bn.device_error(clear=True) == 0
