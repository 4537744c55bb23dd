"""Step-loop parity of the CUDA library against the oracle (Algorithm 1 batched over rows)."""
import numpy as np
import pytest

import rsd_inputs as ri
from helpers import build_pair, parity_step, compare_counters, compare_state

pytestmark = pytest.mark.gpu

TINY = (ri.SHAPES["tiny_draft"], ri.SHAPES["tiny_draft"], ri.SHAPES["tiny_target"])
MINI = (ri.SHAPES["mini_draft"], ri.SHAPES["mini_draft"], ri.SHAPES["mini_target"])
# fp32 path: fp32 sums against fp64 sums; 16-bit path: the bounds asked of bf16 arithmetic
TOL32 = dict(tol_logits=2e-4, tol_reward=1e-5, margin_tok=1e-3, margin_gate=1e-4)
TOL16 = dict(tol_logits=3e-2, tol_reward=1e-2, margin_tok=5e-2, margin_gate=1e-2)


def test_tiny_fp32_config_all_deltas():
    """Tiny fp32 models, batch 4, 64-token prompts, step ends at id 13 or after 32 tokens, 4 steps,
    greedy; delta = 0.7 as configured, plus the median reward (both branches) and the two limits."""
    prompts = ri.prompts(0, 4, 64, 64, 1024)
    base = dict(max_step_tokens=32, max_steps=4, max_seq_tokens=64 + 4 * 32, step_end_id=13, temperature=0.0, seed=0)
    eng, loop = build_pair(TINY, bf16=False, prompts=prompts, loop_kwargs=base)
    compare_state(eng, loop)
    r0 = loop.step(0.0)["rewards"]
    median = float(np.median(r0))
    for delta in (0.7, median, 0.0, 1.5):
        eng, loop = build_pair(TINY, bf16=False, prompts=prompts, loop_kwargs=base)
        stats = {}
        n_acc = 0
        for _ in range(4):
            g, o = parity_step(eng, loop, delta, stats=stats, **TOL32)
            n_acc += int(g["accept"].sum())
        compare_counters(eng, loop)
        assert stats["tokens_compared"] >= 0.9 * stats["tokens"]
        if delta == 0.0:
            assert n_acc == 16 and eng.counters()["gen_tokens"][2] == 0
        if delta == 1.5:
            assert n_acc == 0 and eng.counters()["gen_tokens"][2] == eng.counters()["gen_tokens"][0]
        assert not g["live"].any()          # four steps were the budget
        eng.close()


def test_tiny_free_running_equals_oracle_when_margins_are_clear():
    """Without forcing, wherever every margin of the oracle's trace is clear the GPU must walk the
    same path by itself: same tokens, gate decisions and integer state."""
    prompts = ri.prompts(5, 3, 9, 30, 1024)
    base = dict(max_step_tokens=12, max_steps=3, max_seq_tokens=96, step_end_id=3, step_end_mod=7,
                temperature=0.7, seed=4)
    eng, loop = build_pair(TINY, bf16=False, prompts=prompts, loop_kwargs=base)
    delta = 0.5
    for _ in range(3):
        o = loop.step(delta)
        margins = [m for key in ("draft_trace", "target_trace") for tr in o[key] if tr for m in tr["margin"]]
        gate_margin = np.abs(o["rewards"][o["step_len"] > 0] - delta).min() if (o["step_len"] > 0).any() else 1.0
        if min(margins) < 1e-3 or gate_margin < 1e-4:
            pytest.skip("a margin of the oracle trace is too small for a free-running comparison")
        g = eng.step(delta)
        assert np.array_equal(g["accept"], o["accept"]) and np.array_equal(g["step_len"], o["step_len"])
        for b in range(3):
            assert g["step_tokens"][b, :o["step_len"][b]].tolist() == list(o["step_tokens"][b])
        compare_state(eng, loop)
    compare_counters(eng, loop)


def test_ragged_steps_eos_and_dead_rows():
    """Ragged prompts, steps of different lengths (delimiter by residue), an EOS id, a row that has
    no room to start, and rows that stop at different times."""
    tokens, offsets = ri.prompts(7, 6, 3, 40, 1024)
    base = dict(max_step_tokens=9, max_steps=5, max_seq_tokens=72, step_end_id=2, step_end_mod=5, eos_id=77,
                temperature=0.7, seed=9)
    # row 5 gets a prompt that leaves no room for a step
    long = np.arange(64, dtype=np.int32)
    tokens = np.concatenate([tokens[:offsets[5]], long]).astype(np.int32)
    offsets = offsets.copy(); offsets[6] = offsets[5] + 64
    eng, loop = build_pair(TINY, bf16=False, prompts=(tokens, offsets), loop_kwargs=base)
    r0 = loop.step(0.0)["rewards"]
    delta = float(np.median(r0[r0 > 0]))
    eng, loop = build_pair(TINY, bf16=False, prompts=(tokens, offsets), loop_kwargs=base)
    lens = set()
    for _ in range(5):
        g, o = parity_step(eng, loop, delta, **TOL32)
        lens.update(g["step_len"].tolist())
        assert g["step_len"][5] == 0 and g["live"][5] == 0
    assert len(lens) > 3
    compare_counters(eng, loop)


@pytest.mark.parametrize("kv_extended", [0, 1])
def test_mini_bf16_models(kv_extended):
    """16-bit weights, head_dim 128, Gumbel-max at T = 0.7, chunked multi-token passes; with the
    16-bit KV cache and with the extended one (values as hi + lo pairs)."""
    prompts = ri.prompts(2, 5, 20, 70, 4096)
    base = dict(max_step_tokens=10, max_steps=3, max_seq_tokens=112, step_end_id=1, step_end_mod=6,
                temperature=0.7, seed=21)
    eng, loop = build_pair(MINI, bf16=True, prompts=prompts, loop_kwargs=base)
    r0 = loop.step(0.0)["rewards"]
    delta = float(np.sort(r0)[1])
    eng, loop = build_pair(MINI, bf16=True, prompts=prompts, loop_kwargs=base,
                           engine_kwargs=dict(max_chunk_tokens=64, kv_extended=kv_extended))
    stats = {}
    for _ in range(3):
        parity_step(eng, loop, delta, stats=stats, **TOL16)
    compare_counters(eng, loop)
    print("mini bf16 parity, kv_extended =", kv_extended, stats)


def test_page_pool_exhaustion_is_an_error_not_a_fault():
    from paper_2501_19324_b200 import RsdError
    prompts = ri.prompts(0, 4, 64, 64, 1024)
    base = dict(max_step_tokens=32, max_steps=4, max_seq_tokens=192, step_end_id=13, temperature=0.0, seed=0)
    sh = ri.SHAPES["tiny_draft"]
    page_bytes = sh.n_layers * 2 * sh.n_kv_heads * 16 * sh.head_dim * 4
    with pytest.raises(RsdError) as e:
        build_pair(TINY, bf16=False, prompts=prompts, loop_kwargs=base,
                   engine_kwargs=dict(kv_bytes=[page_bytes * 10, page_bytes * 400, page_bytes * 800]))
    assert e.value.code == -3


@pytest.mark.parametrize("omega_kind,delta,alpha", [(0, 0.6, 0.0), (2, 0.0, 0.0), (3, 0.0, 0.0), (4, 0.5, 30.0)])
def test_general_acceptance_criterion_on_gpu(omega_kind, delta, alpha):
    """Algorithm 2 with the other weighting functions of Table 1 (constant, clip, r/(1+r), logistic):
    the GPU draws the same Philox uniform per (row, |z_i|) and takes the same decision as the oracle."""
    prompts = ri.prompts(11, 8, 10, 24, 1024)
    base = dict(max_step_tokens=6, max_steps=4, max_seq_tokens=64, step_end_id=3, step_end_mod=4,
                temperature=0.7, seed=17, omega_kind=omega_kind, omega_b=alpha)
    eng, loop = build_pair(TINY, bf16=False, prompts=prompts, loop_kwargs=base,
                           engine_kwargs=dict(omega_kind=omega_kind, omega_alpha=alpha))
    seen = set()
    for _ in range(4):
        tol = dict(TOL32, margin_gate=0.0)            # never force the gate: it must agree by itself
        g, o = parity_step(eng, loop, delta, **tol)
        seen.update(g["accept"][g["step_len"] > 0].tolist())
    assert seen == {0, 1}                             # both outcomes occurred
    compare_counters(eng, loop)


def test_reset_and_new_batch_sizes_reuse_one_context():
    """rsd_reset / a second rsd_prefill with another batch size on the same context: pages return to the
    pool, the captured decode graphs are rebuilt for the new slot count, results match a fresh oracle."""
    from oracle.rsd_loop import OracleRSD
    base = dict(max_step_tokens=6, max_steps=3, max_seq_tokens=64, step_end_id=5, step_end_mod=9, temperature=0.7, seed=8)
    p4 = ri.prompts(21, 4, 8, 20, 4096)
    eng, loop = build_pair(MINI, bf16=True, prompts=p4, loop_kwargs=base, engine_kwargs=dict(max_batch=6))
    for _ in range(2):
        parity_step(eng, loop, 0.45, **TOL16)
    for seed, B in ((22, 6), (23, 2)):
        tokens, offsets = ri.prompts(seed, B, 8, 20, 4096)
        eng.prefill(tokens, offsets)                     # drops the old rows
        assert eng.counters()["steps"] == 0
        loop = OracleRSD(*loop.models, loop.cfg)
        loop.prefill([tokens[offsets[b]:offsets[b + 1]].tolist() for b in range(B)])
        compare_state(eng, loop)
        for _ in range(2):
            parity_step(eng, loop, 0.45, **TOL16)
        compare_counters(eng, loop)


def test_call_order_and_argument_errors():
    from paper_2501_19324_b200 import Engine, Model, RsdError
    sh = ri.SHAPES["tiny_draft"]
    models = [Model(sh, ri.gpu_model_tensors(sh, slot, 0, False, hk), hk)
              for slot, hk in enumerate((ri.HEAD_LM, ri.HEAD_REWARD_SIGMOID, ri.HEAD_LM))]
    eng = Engine(*models, max_batch=2, max_seq_tokens=48, max_step_tokens=8, max_steps=2, step_end_id=13)
    eng.B = 2
    with pytest.raises(RsdError) as e:
        eng.step(0.5)                                    # step before prefill
    assert e.value.code == -2
    with pytest.raises(RsdError) as e:
        eng.prefill(np.array([1, 2, 5000], np.int32), np.array([0, 2, 3], np.int32))    # id beyond the vocabulary
    assert e.value.code == -1
    with pytest.raises(RsdError) as e:
        eng.prefill(np.arange(6, dtype=np.int32), np.array([0, 2, 4, 6], np.int32))      # more rows than max_batch
    assert e.value.code == -1
    eng.prefill(np.array([1, 2, 3, 4], np.int32), np.array([0, 2, 4], np.int32))          # still usable afterwards
    r = eng.step(0.0)
    assert r["accept"].all() and (r["step_len"] > 0).all()
    with pytest.raises(RsdError):                        # a PRM must not carry an lm head, and vice versa
        Engine(models[0], models[0], models[2], max_batch=2, max_seq_tokens=48, max_step_tokens=8, max_steps=2, step_end_id=13)
    # models are loaded once per context: the captured decode graphs hold their pointers
    from paper_2501_19324_b200 import lib
    assert lib().rsd_load_models(eng.ctx, models[0].desc, models[1].desc, models[2].desc) == -2
    assert b"once per context" in lib().rsd_last_error(eng.ctx)
    r = eng.step(0.0)                                    # the refusal left the context as it was
    assert (r["step_len"] > 0).all()
    with pytest.raises(RsdError) as e:                   # kv_extended takes 0 (by depth), 1 or 2
        Engine(*models, max_batch=2, max_seq_tokens=48, max_step_tokens=8, max_steps=2, step_end_id=13, kv_extended=3)
    assert e.value.code == -1


@pytest.mark.parametrize("delta,min_rows", [(0.47, 3), (0.49, 4)])
def test_queued_rejections_match_the_oracle(delta, min_rows):
    """rsd_step_queued: rejected rows wait until min_rows wait, then one target pass serves all of
    them.  Compared call by call with the oracle under the same rule (tokens, rewards, gate, waiting
    flags, cursors, page tables, the list of waiting rows, counters), and at the end every row's
    sequence equals the one the lock-step oracle loop writes."""
    shapes = (ri.SHAPES["tiny_draft"], ri.SHAPES["tiny_draft"], ri.SHAPES["tiny_target"])
    prompts = ri.prompts(31, 6, 5, 20, 1024)
    # thresholds just under the tiny PRM's reward range (0.5 +- 0.08): a rejection every few steps
    kw = dict(max_step_tokens=6, max_steps=6, max_seq_tokens=96, step_end_id=3, step_end_mod=5, temperature=0.7, seed=4)
    eng, loop = build_pair(shapes, bf16=False, prompts=prompts, loop_kwargs=kw)
    _, lock = build_pair(shapes, bf16=False, prompts=prompts, loop_kwargs=kw)
    stats = {}
    waited = flushed = 0
    for _ in range(40):
        if not any(r.live for r in loop.rows):
            break
        g, o = parity_step(eng, loop, delta, tol_logits=2e-4, tol_reward=1e-5, margin_tok=1e-3, margin_gate=1e-4,
                           stats=stats, min_target_rows=min_rows)
        waited += int(o["waiting"].sum())
        flushed += int(o["flushed"])
    assert not any(r.live for r in loop.rows)
    assert waited > 0 and flushed > 0
    compare_counters(eng, loop)
    while any(r.live for r in lock.rows):
        lock.step(delta)
    assert [r.z for r in loop.rows] == [r.z for r in lock.rows]
    print("queued rejections, min_rows", min_rows, stats)


def test_queued_with_min_rows_one_is_rsd_step_and_bad_arguments():
    from paper_2501_19324_b200 import lib
    shapes = (ri.SHAPES["tiny_draft"], ri.SHAPES["tiny_draft"], ri.SHAPES["tiny_target"])
    prompts = ri.prompts(32, 4, 5, 12, 1024)
    kw = dict(max_step_tokens=5, max_steps=3, max_seq_tokens=64, step_end_id=3, temperature=0.7, seed=5)
    a, _ = build_pair(shapes, bf16=False, prompts=prompts, loop_kwargs=kw)
    b, _ = build_pair(shapes, bf16=False, prompts=prompts, loop_kwargs=kw)
    for _ in range(3):
        ra = a.step(0.5)
        out = {k: np.zeros_like(v) for k, v in ra.items()}
        ptr = [out[k].ctypes.data for k in ("step_tokens", "step_len", "rewards", "accept", "live", "waiting")]
        assert lib().rsd_step_queued(b.ctx, 0.5, 1, None, *ptr) == 0
        for k in ("step_tokens", "step_len", "rewards", "accept", "live"):
            assert np.array_equal(ra[k], out[k]), k
        assert not out["waiting"].any()
    assert lib().rsd_step_queued(b.ctx, 0.5, 0, None, *ptr) == -1
    assert b"min_target_rows" in lib().rsd_last_error(b.ctx)


@pytest.mark.parametrize("shapes,bf16,tol", [(TINY, False, TOL32), (MINI, True, TOL16)])
def test_merged_prm_on_the_drafts_trunk(shapes, bf16, tol):
    """prm_shares_draft: the reward comes from one more single-token pass of the draft and the PRM's head;
    step-by-step parity with the oracle in the same mode (rewards, gate, tokens, cursors -- the PRM's stay
    at zero -- pages, counters)."""
    prompts = ri.prompts(41, 5, 6, 30, shapes[0].vocab)
    kw = dict(max_step_tokens=6, max_steps=4, max_seq_tokens=96, step_end_id=3, step_end_mod=5, temperature=0.7,
              seed=6, prm_shares_draft=True)
    eng, loop = build_pair(shapes, bf16=bf16, prompts=prompts, loop_kwargs=kw)
    probe = loop.step(0.0)["rewards"]
    delta = float(np.median(probe))
    eng, loop = build_pair(shapes, bf16=bf16, prompts=prompts, loop_kwargs=kw)
    stats, seen = {}, set()
    for _ in range(4):
        g, o = parity_step(eng, loop, delta, stats=stats, **tol)
        seen |= set(int(a) for a, n in zip(o["accept"], o["step_len"]) if n)
    assert seen == {0, 1}
    st = eng.state()
    assert not st["kv_len"][1].any() and not st["n_pages"][1].any()
    compare_counters(eng, loop)
    print("merged PRM", "bf16" if bf16 else "fp32", stats)


@pytest.mark.parametrize("B,ext", [(5, 0), (20, 0), (40, 0), (6, 1)])
def test_persistent_decode_kernel_against_the_oracle_and_the_separate_kernels(B, ext):
    """RSD_DEBUG_PERSISTENT_DECODE: bf16 models at up to 64 rows decode with one persistent kernel per iteration
    (all layers, grid barriers between the phases).  It must meet the oracle like the default kernel-by-kernel
    path, agree with that path far inside the bf16 bound, and launch far fewer kernels.  Batch sizes cover the 16-, 32- and 64-row
    operand tiles; ext = hi + lo KV cache."""
    from paper_2501_19324_b200 import lib, RSD_DEBUG_KEEP_LOGITS, RSD_DEBUG_PERSISTENT_DECODE
    from oracle.rsd_loop import DRAFT, TARGET
    prompts = ri.prompts(50 + B, B, 5, 40, MINI[0].vocab)
    kw = dict(max_step_tokens=5, max_steps=3, max_seq_tokens=80, step_end_id=3, step_end_mod=5, temperature=0.7, seed=8)
    probe_eng, probe = build_pair(MINI, bf16=True, prompts=prompts, loop_kwargs=kw,
                                  engine_kwargs=dict(debug_flags=RSD_DEBUG_KEEP_LOGITS))
    delta = float(np.median(probe.step(0.0)["rewards"]))
    probe_eng.close()
    runs = {}
    for name, flags in (("mega", RSD_DEBUG_KEEP_LOGITS | RSD_DEBUG_PERSISTENT_DECODE), ("separate", RSD_DEBUG_KEEP_LOGITS)):
        eng, loop = build_pair(MINI, bf16=True, prompts=prompts, loop_kwargs=kw,
                               engine_kwargs=dict(debug_flags=flags, kv_extended=ext))
        before = lib().rsd_debug_launch_count()
        stats, logits, seen = {}, [], set()
        for _ in range(3):
            g, o = parity_step(eng, loop, delta, stats=stats, **TOL16)
            seen |= set(int(a) for a, n in zip(o["accept"], o["step_len"]) if n)
            logits.append((eng.logits(DRAFT).copy(), eng.logits(TARGET).copy(), o))
        compare_counters(eng, loop)
        runs[name] = dict(stats=stats, logits=logits, launches=lib().rsd_debug_launch_count() - before, seen=seen)
        eng.close()
    assert runs["mega"]["seen"] == {0, 1}                      # both models decoded
    assert runs["mega"]["launches"] < 0.6 * runs["separate"]["launches"]
    worst = 0.0
    for (d0, t0, o), (d1, t1, _) in zip(runs["mega"]["logits"], runs["separate"]["logits"]):
        for key, a, b in (("draft_trace", d0, d1), ("target_trace", t0, t1)):
            for r in range(B):
                if o[key][r] is not None:
                    n = len(o[key][r]["logits"])
                    worst = max(worst, float(np.abs(a[r, :n] - b[r, :n]).max()))
    assert worst <= 2e-3, worst
    print("persistent decode kernel", B, ext, runs["mega"]["stats"], "vs separate kernels", worst,
          "launches", runs["mega"]["launches"], runs["separate"]["launches"])


def test_persistent_decode_kernel_phase_timeline():
    """rsd_debug_mega_profile: with RSD_DEBUG_MEGA_PROFILE the persistent kernel's first CTA stamps the global timer
    at its start, before and after each of its 7 * layers grid barriers and at its end, in order; without the flag
    the call is refused."""
    from paper_2501_19324_b200 import RSD_DEBUG_KEEP_LOGITS, RSD_DEBUG_PERSISTENT_DECODE, RSD_DEBUG_MEGA_PROFILE
    from paper_2501_19324_b200.binding import RsdError
    from oracle.rsd_loop import DRAFT, TARGET
    prompts = ri.prompts(77, 4, 5, 20, MINI[0].vocab)
    kw = dict(max_step_tokens=3, max_steps=2, max_seq_tokens=48, step_end_id=3, temperature=0.7, seed=2)
    eng, loop = build_pair(MINI, bf16=True, prompts=prompts, loop_kwargs=kw,
                           engine_kwargs=dict(debug_flags=RSD_DEBUG_KEEP_LOGITS | RSD_DEBUG_PERSISTENT_DECODE | RSD_DEBUG_MEGA_PROFILE))
    parity_step(eng, loop, 2.0, **TOL16)                   # delta above the reward range: both models decode
    for which, shape in ((DRAFT, MINI[0]), (TARGET, MINI[2])):
        st = eng.mega_profile(which).astype(np.int64)
        assert len(st) == 14 * shape.n_layers + 2, len(st)
        assert (np.diff(st) >= 0).all() and st[-1] > st[0]
        assert st[-1] - st[0] < 50_000_000                 # one launch of a two- or three-layer model: far below 50 ms
    eng.close()
    eng, loop = build_pair(MINI, bf16=True, prompts=prompts, loop_kwargs=kw)
    with pytest.raises(RsdError):
        eng.mega_profile(DRAFT)
    eng.close()


@pytest.mark.parametrize("shapes,bf16,tol,k", [(TINY, False, TOL32, 3), (MINI, True, TOL16, 4), (TINY, False, TOL32, 1)])
def test_speculative_decoding_of_rejected_steps(shapes, bf16, tol, k):
    """sd_tokens = k (the paper's discussion of combining RSD with speculative decoding): the steps of rejected rows
    are written in rounds of k draft proposals and one target pass.  Step by step against the oracle in the same
    mode: logits of every written token, tokens, cursors of all three caches (the draft's now follow the target's),
    pages, the rounds' counters; and the committed sequences equal those of the plain loop."""
    prompts = ri.prompts(61, 6, 6, 30, shapes[0].vocab)
    kw = dict(max_step_tokens=7, max_steps=4, max_seq_tokens=96, step_end_id=3, step_end_mod=5, temperature=0.7,
              seed=6, sd_tokens=k)
    eng, loop = build_pair(shapes, bf16=bf16, prompts=prompts, loop_kwargs=kw)
    delta = float(np.median(loop.step(0.0)["rewards"]))
    eng, loop = build_pair(shapes, bf16=bf16, prompts=prompts, loop_kwargs=kw)
    _, plain = build_pair(shapes, bf16=bf16, prompts=prompts, loop_kwargs=dict(kw, sd_tokens=0))
    stats, seen = {}, set()
    for _ in range(4):
        g, o = parity_step(eng, loop, delta, stats=stats, **tol)
        seen |= set(int(a) for a, n in zip(o["accept"], o["step_len"]) if n)
        plain.step(delta)
    assert seen == {0, 1}
    assert [r.z for r in loop.rows] == [r.z for r in plain.rows]
    compare_counters(eng, loop)
    c = eng.counters()
    assert c["sd_rounds"] > 0 and c["sd_verified"] == c["sd_proposed"] >= c["gen_tokens"][2]
    print("speculative decoding of rejected steps, k =", k, stats, {q: c[q] for q in c if q.startswith("sd_")})
    eng.close()


@pytest.mark.parametrize("extra,min_rows", [(dict(), 3), (dict(prm_shares_draft=True), 1)])
def test_speculative_decoding_with_queued_rows_and_with_a_merged_prm(extra, min_rows):
    """sd_tokens together with the other two scheduling modes: rejected rows that wait for a shared target pass
    (rsd_step_queued), and a PRM that is a head on the draft's trunk (its scoring pass leaves one more position in
    the draft's cache beyond the cursor, which the proposals then overwrite)."""
    prompts = ri.prompts(63, 6, 5, 20, 1024)
    kw = dict(max_step_tokens=6, max_steps=5, max_seq_tokens=96, step_end_id=3, step_end_mod=5, temperature=0.7,
              seed=12, sd_tokens=3, **extra)
    eng, loop = build_pair(TINY, bf16=False, prompts=prompts, loop_kwargs=kw)
    delta = float(np.median(loop.step(0.0)["rewards"]))
    eng, loop = build_pair(TINY, bf16=False, prompts=prompts, loop_kwargs=kw)
    served = 0
    for _ in range(12):
        if not any(r.live for r in loop.rows):
            break
        g, o = parity_step(eng, loop, delta, min_target_rows=min_rows, **TOL32)
        served += sum(1 for r in o["sd_rounds"] if r)
    assert served > 0
    compare_counters(eng, loop)
    eng.close()


def test_speculative_rounds_keep_the_matching_prefix_on_gpu():
    """Proposals planted around the target's true continuation (known from a first, plain run of the oracle): all
    right, wrong at once, right-right-wrong, a short last round.  The GPU must write the matching prefix plus the
    target's own token, round by round: tokens, cursors and the round counters against the oracle's."""
    from oracle.rsd_loop import OracleRSD, LoopConfig
    shapes = TINY
    prompts = ri.prompts(62, 3, 5, 12, shapes[0].vocab)
    kw = dict(max_step_tokens=9, max_steps=1, max_seq_tokens=40, step_end_id=1 << 20, temperature=0.7, seed=5, sd_tokens=4)
    _, probe = build_pair(shapes, bf16=False, prompts=prompts, loop_kwargs=dict(kw, sd_tokens=0))
    truth = [list(y) for y in probe.step(2.0)["step_tokens"]]          # delta above the range: the target's steps
    bad = lambda t: (t + 1) % 1024
    planted = []
    for b in range(3):
        t = truth[b]
        planted.append([t[0:4], [bad(t[4]), 7, 7, 7], [t[5], t[6], bad(t[7]), t[8]], [t[8]]])
    planted[2] = None                                                   # row 2 keeps the draft's own proposals
    eng, loop = build_pair(shapes, bf16=False, prompts=prompts, loop_kwargs=kw)
    o = loop.step(2.0, forced_sd_props=planted)
    eng.force_tokens(0, o["draft_tokens"])
    eng.force_tokens(2, o["target_tokens"])
    eng.force_sd_proposals([None if r is None else [rd["props"] for rd in r] for r in o["sd_rounds"]])
    g = eng.step(2.0)
    for b in range(3):
        assert g["step_tokens"][b].tolist() == truth[b] == list(o["step_tokens"][b])
    for b in range(2):
        assert [(rd["emitted"], rd["matched"]) for rd in o["sd_rounds"][b]] == [(4, 4), (1, 0), (3, 2), (1, 1)]
    from helpers import compare_state
    compare_state(eng, loop)
    compare_counters(eng, loop)
    smp = eng.sampled(2)
    for b in range(3):                                   # the target's own choices were the truth everywhere
        clear = [j for j in range(9) if o["target_trace"][b]["margin"][j] > 1e-3]
        assert [smp[b, j] for j in clear] == [truth[b][j] for j in clear]
    eng.close()


def test_device_outputs_and_target_step_rewards():
    """rsd_step_device fills device arrays with what rsd_step returns on the host, and the reward of a step the
    target wrote shows up one call later (the PRM caches that step before it scores the next draft step): NaN
    before, equal to the oracle's value afterwards."""
    prompts = ri.prompts(71, 5, 6, 20, 1024)
    kw = dict(max_step_tokens=6, max_steps=4, max_seq_tokens=64, step_end_id=3, step_end_mod=5, temperature=0.7, seed=9)
    a, loop = build_pair(TINY, bf16=False, prompts=prompts, loop_kwargs=kw)
    b, _ = build_pair(TINY, bf16=False, prompts=prompts, loop_kwargs=kw)
    assert np.isnan(a.target_step_rewards()).all()
    delta = float(np.median(loop.step(0.0)["rewards"]))
    _, loop = build_pair(TINY, bf16=False, prompts=prompts, loop_kwargs=kw)
    seen = 0
    for i in range(4):
        o = loop.step(delta)
        host = a.step(delta)
        dev = b.step_device(delta)
        for k in ("step_tokens", "step_len", "rewards", "accept", "live"):
            assert np.array_equal(host[k], dev[k].cpu().numpy()), k
        fresh = ~np.isnan(o["target_rewards"])
        got = a.target_step_rewards()
        if fresh.any():
            assert np.abs(got[fresh] - o["target_rewards"][fresh]).max() <= 1e-5
            seen += int(fresh.sum())
        if i == 0:
            assert np.isnan(got).all()                                   # nothing the target wrote has been scored yet
    assert seen > 0
    a.close(); b.close()


def test_batches_of_more_than_64_rows_and_wide_heads():
    """65 to 128 rows: K-split products over the whole machine, and the persistent kernel for the gate/up and the head with
    more weight tiles than SMs (RMSNorm denominators and idle flag included), against the oracle."""
    from dataclasses import replace
    d, t = (replace(s, vocab=19300, d_ffn=9600) for s in (MINI[0], MINI[2]))
    prompts = ri.prompts(93, 100, 2, 6, d.vocab)
    base = dict(max_step_tokens=2, max_steps=2, max_seq_tokens=16, step_end_id=3, step_end_mod=5, temperature=0.7, seed=9)
    eng, loop = build_pair((d, d, t), bf16=True, prompts=prompts, loop_kwargs=base)
    stats = {}
    parity_step(eng, loop, 2.0, stats=stats, **TOL16)          # every row is rejected: the target decodes 100 rows too
    assert stats["tokens_compared"] > 0.5 * stats["tokens"]
    compare_counters(eng, loop)
    eng.close()


@pytest.mark.parametrize("d,H,KV,hd,ext", [(128, 1, 1, 64, 0), (512, 7, 1, 128, 0), (2048, 8, 1, 64, 0), (512, 8, 2, 64, 1), (512, 8, 1, 128, 1)])
def test_decode_attention_that_takes_the_qkv_product(d, H, KV, hd, ext):
    """Contexts in one split: the attention adds up the product's K splits (1, 4 and 16 of them), rotates and writes the cache
    itself; head groups of one to eight, both head sizes, a new token on the first and the last place of a page."""
    sh = ri.ModelShape(2, d, H, KV, hd, 512, 1024)
    prompts = ri.prompts(31 + H, 5, 13, 18, sh.vocab)
    kw = dict(max_step_tokens=6, max_steps=2, max_seq_tokens=48, step_end_id=3, step_end_mod=7, temperature=0.7, seed=4)
    eng, loop = build_pair((sh, sh, sh), bf16=True, prompts=prompts, loop_kwargs=kw, engine_kwargs=dict(kv_extended=ext))
    stats = {}
    for _ in range(2):
        parity_step(eng, loop, 2.0, stats=stats, **TOL16)      # every row is rejected: draft and target decode
    assert stats["tokens_compared"] > 0.5 * stats["tokens"]
    eng.close()


@pytest.mark.parametrize("d,H,KV,hd,lo,hi", [(256, 4, 2, 64, 10, 20), (512, 4, 1, 128, 250, 270)])
def test_fp32_caches_may_start_anywhere(monkeypatch, d, H, KV, hd, lo, hi):
    """fp32 pools that start 4 bytes off a 16-byte boundary, read element by element, give the same steps: the decode attention with the
    rotation inside, a new token on the first and last place of a page, fewer pages than warps and more."""
    import torch
    from paper_2501_19324_b200 import Engine, Model
    sh = ri.ModelShape(2, d, H, KV, hd, 344, 1024)
    heads = (ri.HEAD_LM, ri.HEAD_REWARD_SIGMOID, ri.HEAD_LM)
    models = [Model(sh, ri.gpu_model_tensors(sh, slot, 0, False, hk), hk) for slot, hk in enumerate(heads)]
    empty, out = torch.empty, []
    for off in (0, 4):
        calls = []

        def placed(*size, **kw):
            calls.append(size)
            if len(calls) > 3:                                  # the three pools come first, then the workspace
                return empty(*size, **kw)
            return empty(size[0] + 16, **kw)[off:off + size[0]]
        monkeypatch.setattr(torch, "empty", placed)
        eng = Engine(*models, max_batch=5, max_seq_tokens=hi + 24, max_step_tokens=8, max_steps=2, step_end_id=-1, temperature=0.7, seed=2)
        monkeypatch.setattr(torch, "empty", empty)
        assert all(eng.cfg.kv_pool[i] % 16 == off for i in range(3))
        eng.prefill(*ri.prompts(5, 5, lo, hi, sh.vocab))
        out.append([eng.step(2.0) for _ in range(2)])
        eng.close()
    for a, b in zip(*out):
        for k in a:
            np.testing.assert_array_equal(a[k], b[k])


def test_16_bit_caches_off_a_boundary_are_refused(monkeypatch):
    """The tensor-core attention copies 16 bytes at a time: a pool 4 bytes off a boundary is refused before anything runs on it."""
    import torch
    from paper_2501_19324_b200 import Engine, Model
    from paper_2501_19324_b200.binding import RsdError
    heads = (ri.HEAD_LM, ri.HEAD_REWARD_SIGMOID, ri.HEAD_LM)
    models = [Model(sh, ri.gpu_model_tensors(sh, slot, 0, True, hk), hk) for slot, (sh, hk) in enumerate(zip(MINI, heads))]
    empty = torch.empty
    monkeypatch.setattr(torch, "empty", lambda *size, **kw: empty(size[0] + 512, **kw)[4:4 + size[0]] if kw["dtype"] == torch.uint8 and size[0] < (8 << 20) else empty(*size, **kw))
    with pytest.raises(RsdError, match="16-byte aligned"):
        Engine(*models, max_batch=2, max_seq_tokens=32, max_step_tokens=4, max_steps=2, step_end_id=3)


@pytest.mark.parametrize("bf16", [False, True])
def test_norm_gains_may_start_anywhere(bf16):
    """Norm gains one element off any wider boundary give the same step."""
    import torch
    from paper_2501_19324_b200 import Engine, Model
    shapes = MINI if bf16 else TINY
    heads = (ri.HEAD_LM, ri.HEAD_REWARD_SIGMOID, ri.HEAD_LM)

    def off(g):
        return torch.cat([g[:1], g])[1:]
    out = []
    for move in (lambda g: g, off):
        models = []
        for slot, (sh, hk) in enumerate(zip(shapes, heads)):
            t = dict(ri.gpu_model_tensors(sh, slot, 0, bf16, hk))
            t.update(final_norm=move(t["final_norm"]), norm1=[move(g) for g in t["norm1"]], norm2=[move(g) for g in t["norm2"]])
            models.append(Model(sh, t, hk))
        eng = Engine(*models, max_batch=3, max_seq_tokens=40, max_step_tokens=6, max_steps=2, step_end_id=3, temperature=0.7, seed=2)
        eng.prefill(*ri.prompts(5, 3, 10, 20, shapes[0].vocab))
        out.append([eng.step(2.0) for _ in range(2)])
        eng.close()
    for a, b in zip(*out):
        for k in a:
            np.testing.assert_array_equal(a[k], b[k])


@pytest.mark.parametrize("d,H,KV,hd,F,rows,ext", [(64, 1, 1, 64, 64, 1, 0), (576, 7, 1, 128, 448, 8, 0), (576, 7, 1, 128, 448, 9, 0), (512, 4, 2, 64, 1408, 5, 1),
                                                  (1536, 12, 2, 128, 1024, 4, 0), (1536, 12, 2, 128, 1024, 6, 0), (512, 8, 8, 128, 520, 2, 1)])
def test_decode_products_of_few_rows(d, H, KV, hd, F, rows, ext):
    """bf16 decode passes of one to eight rows and one more, products with their next step and (wide shapes, more rows; K off a multiple of
    64) K splits side by side: sums of squares per 8 and per 256 columns, one chunk of K a warp and several, both head sizes,
    both caches, a new token on the first and last place of a page."""
    sh = ri.ModelShape(2, d, H, KV, hd, F, 1024)
    prompts = ri.prompts(11 + d, rows, 14, 18, sh.vocab)
    kw = dict(max_step_tokens=6, max_steps=2, max_seq_tokens=48, step_end_id=3, step_end_mod=7, temperature=0.7, seed=4)
    eng, loop = build_pair((sh, sh, sh), bf16=True, prompts=prompts, loop_kwargs=kw, engine_kwargs=dict(kv_extended=ext))
    stats = {}
    for _ in range(2):
        parity_step(eng, loop, 2.0, stats=stats, **TOL16)      # every row is rejected: draft and target decode
    assert stats["tokens_compared"] > 0.4 * stats["tokens"]
    eng.close()


@pytest.mark.parametrize("d,H,KV,hd,rows,lo,hi", [(64, 1, 1, 64, 3, 13, 18), (260, 4, 2, 128, 9, 14, 33), (128, 10, 1, 64, 5, 252, 262)])
def test_fp32_decode_with_the_small_steps_inside_the_products(d, H, KV, hd, rows, lo, hi):
    """fp32 decode passes: norms and SwiGLU in the products, rotation and page write in the attention; one head group and groups of
    ten, both head sizes, more rows than a block of the product takes, a new token on the first and last place of a page, more
    pages than warps."""
    sh = ri.ModelShape(2, d, H, KV, hd, 344, 1024)
    prompts = ri.prompts(7 + d, rows, lo, hi, sh.vocab)
    kw = dict(max_step_tokens=8, max_steps=2, max_seq_tokens=hi + 24, step_end_id=3, step_end_mod=9, temperature=0.7, seed=4)
    eng, loop = build_pair((sh, sh, sh), bf16=False, prompts=prompts, loop_kwargs=kw)
    stats = {}
    for _ in range(2):
        parity_step(eng, loop, 2.0, stats=stats, **TOL32)      # every row is rejected: draft and target decode
    assert stats["tokens_compared"] > 0.9 * stats["tokens"]
    eng.close()


@pytest.mark.parametrize("bf16,rows", [(False, 3), (True, 2), (True, 9)])
def test_timed_decode_products_count_the_same_bytes(bf16, rows):
    """The bytes reported with the timed products of a decode iteration are the algorithm's: weights and input once, output once or, added
    to, twice.  They don't depend on the kernels that run (of few bf16 rows, of more, fp32); a fused gate/up writes F columns, in bf16
    as pairs in and out."""
    from paper_2501_19324_b200 import Engine, Model
    sh = (MINI if bf16 else TINY)[0]
    heads = (ri.HEAD_LM, ri.HEAD_REWARD_SIGMOID, ri.HEAD_LM)
    models = [Model(sh, ri.gpu_model_tensors(sh, slot, 0, bf16, hk), hk, head_only=slot == 1) for slot, hk in enumerate(heads)]
    eng = Engine(*models, max_batch=rows, max_seq_tokens=48, max_step_tokens=6, max_steps=2, step_end_id=-1, temperature=0.0, prm_shares_draft=1)
    eng.prefill(*ri.prompts(3, rows, 10, 20, sh.vocab))
    eng.gemm_timing(1 << 20)                  # of multi-token passes one in a million, of decode iterations the sixth
    eng.step(-1.0)                            # every row is accepted: the draft alone decodes
    got = eng.gemm_timing(0)
    d, F, T, e = sh.d_model, sh.d_ffn, rows, 2 if bf16 else 4
    width, wide = (sh.n_heads + 2 * sh.n_kv_heads) * sh.head_dim, sh.n_heads * sh.head_dim

    def product(N, K, adds=False):
        return (N + T) * K * e + T * N * (8 if adds else 4)
    layer = product(width, d) + product(d, wide, True) + product(d, F, True)
    layer += 2 * F * d * e + (2 * T * d * e + 2 * T * F * e if bf16 else T * (d + F) * e)
    assert got["launches"] == 4 * sh.n_layers + 1
    assert got["bytes"] == sh.n_layers * layer + product(sh.vocab, d)
    eng.close()


@pytest.mark.parametrize("rows,H,KV,hd,lo,hi", [(97, 1, 1, 64, 3, 18), (37, 16, 4, 128, 12, 33), (74, 14, 2, 128, 12, 20), (100, 8, 1, 128, 250, 262)])
def test_decode_attention_of_sixteen_warps(rows, H, KV, hd, lo, hi):
    """97 to 148 (slot, KV head) pairs: one CTA of sixteen warps each takes the qkv product; groups of one to eight heads, both head
    sizes, fewer pages than warps and more."""
    sh = ri.ModelShape(2, 512, H, KV, hd, 512, 1024)
    prompts = ri.prompts(29 + H, rows, lo, hi, sh.vocab)
    kw = dict(max_step_tokens=4, max_steps=1, max_seq_tokens=hi + 8, step_end_id=3, step_end_mod=7, temperature=0.7, seed=4)
    eng, loop = build_pair((sh, sh, sh), bf16=True, prompts=prompts, loop_kwargs=kw)
    stats = {}
    parity_step(eng, loop, 2.0, stats=stats, **TOL16)          # every row is rejected: draft and target decode
    assert stats["tokens_compared"] > 0.4 * stats["tokens"]
    eng.close()


# One launch per decode phase: the smallest and the widest models that it takes, columns that do not fill the last stage (512 / 256) or the
# last unit of the head, groups of one to eight heads, contexts of one page to three rounds of the warps, one to eight rows.
RESIDENT = [
    # shape, bf16, rows, prompt tokens, extended cache
    (ri.ModelShape(1, 64, 1, 1, 128, 64, 515), True, 1, (3, 3), 0),
    (ri.ModelShape(3, 192, 3, 3, 128, 320, 1000), True, 5, (1, 40), 0),
    (ri.ModelShape(2, 512, 4, 2, 128, 1408, 4096), True, 8, (120, 300), 0),
    (ri.ModelShape(2, 512, 4, 2, 128, 1408, 4096), True, 3, (120, 300), 1),
    (ri.ModelShape(2, 1024, 16, 2, 128, 2048, 1030), True, 7, (10, 150), 0),
    (ri.ModelShape(1, 2048, 8, 8, 128, 1088, 1030), True, 4, (10, 50), 1),
    (ri.ModelShape(1, 16, 1, 1, 64, 8, 100), False, 2, (1, 5), 0),
    (ri.ModelShape(2, 336, 5, 5, 64, 200, 333), False, 8, (3, 70), 0),
    (ri.ModelShape(2, 256, 4, 2, 64, 688, 1024), False, 4, (100, 300), 0),
    (ri.ModelShape(1, 2048, 32, 2, 64, 2048, 520), False, 5, (10, 40), 0),
]


@pytest.mark.parametrize("sh,bf16,rows,ctx,ext", RESIDENT)
def test_decode_phase_in_one_launch(sh, bf16, rows, ctx, ext):
    from paper_2501_19324_b200 import lib, RSD_DEBUG_KEEP_LOGITS
    from paper_2501_19324_b200.binding import RSD_DEBUG_RESIDENT_LOGITS
    prompts = ri.prompts(61 + rows, rows, *ctx, sh.vocab)
    kw = dict(max_step_tokens=7, max_steps=3, max_seq_tokens=ctx[1] + 32, step_end_id=2, step_end_mod=5, temperature=0.7, seed=6)
    launches = []
    for flags in (RSD_DEBUG_KEEP_LOGITS | RSD_DEBUG_RESIDENT_LOGITS, RSD_DEBUG_KEEP_LOGITS):
        eng, loop = build_pair((sh, sh, sh), bf16=bf16, prompts=prompts, loop_kwargs=kw, engine_kwargs=dict(debug_flags=flags, kv_extended=ext))
        stats = {}
        before = lib().rsd_debug_launch_count()
        for _ in range(2):
            parity_step(eng, loop, 2.0, stats=stats, **(TOL16 if bf16 else TOL32))    # every row is rejected: draft and target decode
        launches.append(lib().rsd_debug_launch_count() - before)
        assert stats["tokens"] > 0
        compare_counters(eng, loop)
        eng.close()
    assert launches[0] < launches[1]

def _shared_memory_full_of_nan():
    """Every SM's shared memory, as far as the rings of the products reach, is left with NaN."""
    import torch
    from paper_2501_19324_b200.binding import k_gemm
    W = torch.full((4 * 148 * 128, 2048), float("nan"), dtype=torch.bfloat16, device="cuda")
    for rows in (32, 64, 128, 512):
        k_gemm(W, W[:rows].clone(), x_lo=W[:rows].clone())
    torch.cuda.synchronize()


@pytest.mark.parametrize("rows", [4, 5, 8])
@pytest.mark.parametrize("sh", [ri.ModelShape(2, 64, 1, 1, 64, 96, 300), ri.ModelShape(1, 128, 2, 2, 64, 128, 333), ri.ModelShape(2, 640, 2, 2, 64, 328, 300)],
                         ids=["64", "128", "640"])
def test_fp32_decode_phase_in_one_launch_reads_what_it_wrote(sh, rows):
    """Products whose columns do not fill the last stage, after a kernel that left NaN in shared memory: the columns beyond the last meet weights of
    zero, and zero times what lies there must be zero."""
    from paper_2501_19324_b200 import RSD_DEBUG_KEEP_LOGITS
    from paper_2501_19324_b200.binding import RSD_DEBUG_RESIDENT_LOGITS
    prompts = ri.prompts(71 + rows, rows, 3, 20, sh.vocab)
    kw = dict(max_step_tokens=5, max_steps=3, max_seq_tokens=52, step_end_id=2, step_end_mod=7, temperature=0.7, seed=8)
    eng, loop = build_pair((sh, sh, sh), bf16=False, prompts=prompts, loop_kwargs=kw,
                           engine_kwargs=dict(debug_flags=RSD_DEBUG_KEEP_LOGITS | RSD_DEBUG_RESIDENT_LOGITS))
    for _ in range(2):
        _shared_memory_full_of_nan()
        _, o = parity_step(eng, loop, 2.0, **TOL32)
        for b in range(rows):
            n = len(o["draft_trace"][b]["sampled"])
            assert np.isfinite(eng.logits(0)[b, :n]).all()
    eng.close()


@pytest.mark.parametrize("H,KV", [(4, 2), (8, 1), (16, 2)])
def test_fp32_decode_phase_in_one_launch_over_its_own_keys(H, KV):
    """A group's new key and value are put into the page by the CTA of its first head and read by those of the others, iteration after iteration of one
    launch: long steps behind short prompts, so that nearly all that is attended was written by the phase itself."""
    from paper_2501_19324_b200 import RSD_DEBUG_KEEP_LOGITS
    from paper_2501_19324_b200.binding import RSD_DEBUG_RESIDENT_LOGITS
    sh = ri.ModelShape(3, 256, H, KV, 64, 344, 500)
    prompts = ri.prompts(5, 3, 2, 4, sh.vocab)
    kw = dict(max_step_tokens=70, max_steps=2, max_seq_tokens=150, step_end_id=-1, temperature=0.7, seed=3)
    eng, loop = build_pair((sh, sh, sh), bf16=False, prompts=prompts, loop_kwargs=kw,
                           engine_kwargs=dict(debug_flags=RSD_DEBUG_KEEP_LOGITS | RSD_DEBUG_RESIDENT_LOGITS))
    stats = {}
    parity_step(eng, loop, 2.0, stats=stats, **TOL32)
    assert stats["tokens"] == 2 * 3 * 70
    eng.close()


@pytest.mark.parametrize("temperature", [0.0, 0.7])
@pytest.mark.parametrize("sh,bf16", [(ri.ModelShape(2, 512, 4, 2, 128, 1408, 4096), True), (ri.ModelShape(4, 512, 8, 2, 64, 1376, 1024), False)], ids=["bf16", "fp32"])
def test_kept_logits_are_those_of_the_tokens(sh, bf16, temperature):
    """Logits kept with RSD_DEBUG_LOGITS_AS_DECODED change nothing: the steps and rewards of a small model are, bit by bit, those without them, and a greedy
    token is the first of the largest logits."""
    from paper_2501_19324_b200 import Engine, Model, RSD_DEBUG_KEEP_LOGITS, RSD_DEBUG_LOGITS_AS_DECODED
    heads = (ri.HEAD_LM, ri.HEAD_REWARD_SIGMOID, ri.HEAD_LM)
    models = [Model(sh, ri.gpu_model_tensors(sh, slot, 0, bf16, hk), hk) for slot, hk in enumerate(heads)]
    tokens, offsets = ri.prompts(44, 5, 5, 60, sh.vocab)
    got = []
    for flags in (0, RSD_DEBUG_KEEP_LOGITS | RSD_DEBUG_LOGITS_AS_DECODED):
        eng = Engine(*models, max_batch=5, max_seq_tokens=160, max_step_tokens=20, max_steps=4, step_end_id=1, step_end_mod=15,
                     temperature=temperature, seed=2, debug_flags=flags)
        eng.prefill(tokens, offsets)
        steps = []
        for delta, which in ((2.0, 2), (0.0, 0), (2.0, 2)):            # every row by the target, none, every row
            r = eng.step(delta)
            steps.append({k: v.tobytes() for k, v in r.items()})
            if flags and temperature == 0.0:
                kept = eng.logits(which)
                for b in range(5):
                    n = r["step_len"][b]
                    assert (kept[b, :n].argmax(1) == r["step_tokens"][b, :n]).all()
        got.append(steps)
        eng.close()
    assert got[0] == got[1]


@pytest.mark.parametrize("sh,bf16", [(ri.ModelShape(2, 512, 4, 2, 128, 1408, 4096), True), (ri.ModelShape(2, 256, 4, 2, 64, 688, 1024), False)], ids=["bf16", "fp32"])
def test_decode_phase_where_one_launch_does_not_fit(sh, bf16):
    """A stream that belongs to a part of the chip cannot hold all the CTAs of the one launch at once: the phase runs kernel by kernel, not at all wrong
    or refused, and in one launch again where there is room."""
    from paper_2501_19324_b200 import lib, RSD_DEBUG_KEEP_LOGITS
    from paper_2501_19324_b200.binding import RSD_DEBUG_RESIDENT_LOGITS
    prompts = ri.prompts(12, 3, 10, 40, sh.vocab)
    kw = dict(max_step_tokens=12, max_steps=4, max_seq_tokens=100, step_end_id=2, step_end_mod=50, temperature=0.7, seed=6)
    eng, loop = build_pair((sh, sh, sh), bf16=bf16, prompts=prompts, loop_kwargs=kw,
                           engine_kwargs=dict(debug_flags=RSD_DEBUG_KEEP_LOGITS | RSD_DEBUG_RESIDENT_LOGITS))
    launches = []
    for sms in (0, 40, 0):
        assert lib().rsd_debug_sm_limit(eng.ctx, sms) == 0
        before = lib().rsd_debug_launch_count()
        parity_step(eng, loop, 2.0, **(TOL16 if bf16 else TOL32))
        launches.append(lib().rsd_debug_launch_count() - before)
    assert launches[1] > 2 * max(launches[0], launches[2])
    eng.close()


@pytest.mark.parametrize("sh,bf16,prompt,one_launch", [
    (ri.ModelShape(2, 512, 4, 2, 128, 1408, 4096), True, 520, [1, 1, 0]),         # bf16, one row: 544 tokens
    (ri.ModelShape(2, 256, 4, 2, 64, 688, 1024), False, 424, [1, 1, 0]),          # fp32, one row: 448
    (ri.ModelShape(1, 256, 2, 1, 128, 704, 7168), True, 20, [1]),                 # a vocabulary of 1024 ids a layer and 6144
    (ri.ModelShape(1, 256, 2, 1, 128, 704, 7176), True, 20, [0]),
    (ri.ModelShape(1, 160, 1, 1, 64, 640, 5535), False, 20, [1]),                 # 64 a column, by the CTAs' share of 148
    (ri.ModelShape(1, 160, 1, 1, 64, 640, 5536), False, 20, [0]),
    (ri.ModelShape(1, 1792, 2, 1, 128, 1216, 300), True, 20, [1]),                # columns
    (ri.ModelShape(1, 1856, 2, 1, 128, 1216, 300), True, 20, [0]),
    (ri.ModelShape(1, 1040, 2, 1, 64, 1200, 300), False, 20, [0]),
    (ri.ModelShape(1, 256, 2, 1, 128, 576, 300), True, 20, [0]),                  # 72 CTAs
    (ri.ModelShape(1, 768, 2, 1, 64, 760, 300), False, 20, [0]),                  # 95, fewer than columns / 8
    (ri.ModelShape(1, 1024, 16, 2, 128, 1152, 300), True, 20, [0]),               # 160 units of qkv for 144
    (ri.ModelShape(1, 192, 1, 1, 128, 768, 300), True, 20, [1]),                  # d_ffn, heads beside the columns
    (ri.ModelShape(1, 192, 1, 1, 128, 832, 300), True, 20, [0]),
    (ri.ModelShape(1, 256, 5, 1, 128, 704, 300), True, 20, [0]),
], ids=["bf16-ctx", "fp32-ctx", "bf16-ids", "bf16-ids+", "fp32-ids", "fp32-ids+", "bf16-wide", "bf16-wide+", "fp32-wide+", "grid", "fp32-grid", "qkv", "ffn", "ffn+", "heads+"])
def test_where_decode_phases_are_one_launch(sh, bf16, prompt, one_launch):
    """On both sides of each line between the one launch and the single kernels, and across it as a row grows."""
    from paper_2501_19324_b200 import lib, RSD_DEBUG_KEEP_LOGITS, RSD_DEBUG_LOGITS_AS_DECODED
    prompts = ri.prompts(15, 1, prompt, prompt, sh.vocab)
    kw = dict(max_step_tokens=12, max_steps=4, max_seq_tokens=prompt + 48, step_end_id=-1, temperature=0.7, seed=6)
    eng, loop = build_pair((sh, sh, sh), bf16=bf16, prompts=prompts, loop_kwargs=kw,
                           engine_kwargs=dict(debug_flags=RSD_DEBUG_KEEP_LOGITS | RSD_DEBUG_LOGITS_AS_DECODED))
    for one in one_launch:
        before = lib().rsd_debug_launch_count()
        parity_step(eng, loop, 2.0, **(TOL16 if bf16 else TOL32))
        assert (lib().rsd_debug_launch_count() - before < 100) == bool(one)       # two phases of 12 iterations, eight kernels or more each
    eng.close()


def test_decode_phases_in_one_launch_on_two_streams():
    """Two contexts, a thread and a stream each: each phase takes the whole chip, and none may wait for a part of it."""
    import threading
    import torch
    prompts = ri.prompts(3, 4, 10, 40, MINI[0].vocab)
    kw = dict(max_seq_tokens=160, max_step_tokens=24, max_steps=4, step_end_id=3, step_end_mod=9, temperature=0.7, seed=1)
    engines = [_engine(prompts, **kw) for _ in range(3)]
    want = [engines[0].step(2.0)["step_tokens"].tolist() for _ in range(4)]
    got, failed = [[], []], []

    def run(i):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(4):
                    got[i].append(engines[i + 1].step(2.0)["step_tokens"].tolist())
        except Exception as e:                           # noqa: BLE001
            failed.append(e)
    threads = [threading.Thread(target=run, args=(i,)) for i in range(2)]
    for th in threads:
        th.start()
    for th in threads:
        th.join()
    assert not failed, failed
    assert got[0] == want and got[1] == want
    for e in engines:
        e.close()


def test_decode_phases_on_a_part_of_the_chip():
    """A stream of a green context with 40 SMs: its phases run kernel by kernel, the default stream's in one launch."""
    import torch
    from paper_2501_19324_b200 import lib, RSD_DEBUG_KEEP_LOGITS
    from paper_2501_19324_b200.binding import RSD_DEBUG_RESIDENT_LOGITS
    drv = pytest.importorskip("cuda.bindings.driver")

    def ok(r):
        assert int(r[0]) == 0, r
        return r[1]
    sm = drv.CUdevResourceType.CU_DEV_RESOURCE_TYPE_SM
    sh = MINI[0]
    prompts = ri.prompts(12, 3, 10, 40, sh.vocab)
    kw = dict(max_step_tokens=12, max_steps=4, max_seq_tokens=100, step_end_id=2, step_end_mod=50, temperature=0.7, seed=6)
    eng, loop = build_pair((sh, sh, sh), bf16=True, prompts=prompts, loop_kwargs=kw,
                           engine_kwargs=dict(debug_flags=RSD_DEBUG_KEEP_LOGITS | RSD_DEBUG_RESIDENT_LOGITS))
    dev = ok(drv.cuDeviceGet(torch.cuda.current_device()))
    part = ok(drv.cuDevSmResourceSplitByCount(1, ok(drv.cuDeviceGetDevResource(dev, sm)), 0, 40))[0]
    green = ok(drv.cuGreenCtxCreate(ok(drv.cuDevResourceGenerateDesc([part], 1)), dev, drv.CUgreenCtxCreate_flags.CU_GREEN_CTX_DEFAULT_STREAM))
    stream = ok(drv.cuGreenCtxStreamCreate(green, drv.CUstream_flags.CU_STREAM_NON_BLOCKING, 0))
    launches = []
    for st in (torch.cuda.current_stream(), torch.cuda.ExternalStream(int(stream)), torch.cuda.current_stream()):
        torch.cuda.synchronize()
        before = lib().rsd_debug_launch_count()
        with torch.cuda.stream(st):
            parity_step(eng, loop, 2.0, **TOL16)
        launches.append(lib().rsd_debug_launch_count() - before)
    torch.cuda.synchronize()
    assert launches[1] > 2 * max(launches[0], launches[2])
    eng.close()
    ok((drv.cuStreamDestroy(stream)[0], None))
    ok((drv.cuGreenCtxDestroy(green)[0], None))


@pytest.mark.parametrize("sh,bf16,rows", [(ri.ModelShape(2, 512, 4, 2, 128, 1408, 4096), True, 8), (ri.ModelShape(1, 2048, 8, 8, 128, 1088, 1030), True, 5),
                                          (ri.ModelShape(4, 512, 8, 2, 64, 1376, 1024), False, 3), (ri.ModelShape(1, 2048, 32, 2, 64, 2048, 520), False, 8)],
                         ids=["bf16", "bf16-wide", "fp32", "fp32-wide"])
def test_decode_phases_in_one_launch_share_the_chip(sh, bf16, rows):
    """Callers that run at the same time get a part of the SMs each, and each CTA more units: the same bits."""
    from paper_2501_19324_b200 import Engine, Model, lib, RSD_DEBUG_KEEP_LOGITS
    from paper_2501_19324_b200.binding import RSD_DEBUG_RESIDENT_LOGITS
    heads = (ri.HEAD_LM, ri.HEAD_REWARD_SIGMOID, ri.HEAD_LM)
    models = [Model(sh, ri.gpu_model_tensors(sh, slot, 0, bf16, hk), hk) for slot, hk in enumerate(heads)]
    prompts = ri.prompts(8, rows, 5, 60, sh.vocab)
    got = []
    for n in (1, 2, 3, 4, 9):
        eng = Engine(*models, max_batch=rows, max_seq_tokens=120, max_step_tokens=9, max_steps=3, step_end_id=1, step_end_mod=30,
                     temperature=0.7, seed=2, debug_flags=RSD_DEBUG_KEEP_LOGITS | RSD_DEBUG_RESIDENT_LOGITS)
        eng.prefill(*prompts)
        assert lib().rsd_debug_step_calls(eng.ctx, n) == 0
        seen = []
        for delta, which in ((2.0, 2), (0.0, 0)):
            r = eng.step(delta)
            kept = eng.logits(which)
            seen.append([v.tobytes() for v in r.values()] + [kept[b, :r["step_len"][b]].tobytes() for b in range(rows)])
        got.append(seen)
        eng.close()
    assert all(g == got[0] for g in got)


def _engine(prompts, **kw):
    from paper_2501_19324_b200 import Engine, Model
    heads = (ri.HEAD_LM, ri.HEAD_REWARD_SIGMOID, ri.HEAD_LM)
    eng = Engine(*[Model(sh, ri.gpu_model_tensors(sh, slot, 0, True, hk), hk) for slot, (sh, hk) in enumerate(zip(MINI, heads))],
                 max_batch=len(prompts[1]) - 1, **kw)
    eng.prefill(*prompts)
    return eng


def test_a_failing_decode_phase_ends_early():
    """The error flag of an expired wait, raised ahead of the fourth of 64 iterations: the call reports it after a few iterations
    more, not after the whole phase, and the context refuses further work."""
    from paper_2501_19324_b200.binding import RsdError, lib
    prompts = ri.prompts(1, 3, 10, 20, MINI[0].vocab)
    eng = _engine(prompts, max_seq_tokens=160, max_step_tokens=64, max_steps=3, step_end_id=-1, temperature=0.7, seed=1)
    before = lib().rsd_debug_launch_count()
    eng.step(0.0)                                       # 64 draft iterations, the target has nothing to do
    whole = lib().rsd_debug_launch_count() - before
    assert lib().rsd_debug_fail_iteration(eng.ctx, 3) == 0
    before = lib().rsd_debug_launch_count()
    with pytest.raises(RsdError) as e:
        eng.step(0.0)
    assert e.value.code == -5
    assert lib().rsd_debug_launch_count() - before < whole / 4
    with pytest.raises(RsdError) as e:
        eng.step(0.0)
    assert e.value.code == -2
    eng.close()


def test_a_failing_decode_phase_of_single_kernels_ends_early():
    """The same where the iterations are launched one by one (small models do that when logits are kept): the host follows the phase and launches a few
    iterations more, not all 64."""
    from paper_2501_19324_b200 import RSD_DEBUG_KEEP_LOGITS
    from paper_2501_19324_b200.binding import RsdError, lib
    prompts = ri.prompts(1, 3, 10, 20, MINI[0].vocab)
    eng = _engine(prompts, max_seq_tokens=160, max_step_tokens=64, max_steps=3, step_end_id=-1, temperature=0.7, seed=1, debug_flags=RSD_DEBUG_KEEP_LOGITS)
    before = lib().rsd_debug_launch_count()
    eng.step(0.0)
    whole = lib().rsd_debug_launch_count() - before
    assert whole > 64 * 8
    assert lib().rsd_debug_fail_iteration(eng.ctx, 3) == 0
    before = lib().rsd_debug_launch_count()
    with pytest.raises(RsdError) as e:
        eng.step(0.0)
    assert e.value.code == -5
    assert lib().rsd_debug_launch_count() - before < whole / 4
    with pytest.raises(RsdError) as e:
        eng.step(0.0)
    assert e.value.code == -2
    eng.close()


def test_a_failing_decode_phase_in_one_launch_ends_early():
    """... and where the phase is one launch: the flag is up ahead of it, and it leaves with the first iteration, whose successors sample nothing."""
    from paper_2501_19324_b200.binding import RsdError, lib
    prompts = ri.prompts(1, 3, 10, 20, MINI[0].vocab)
    eng = _engine(prompts, max_seq_tokens=160, max_step_tokens=64, max_steps=3, step_end_id=-1, temperature=0.7, seed=1)
    before = lib().rsd_debug_launch_count()
    eng.step(0.0)
    assert lib().rsd_debug_launch_count() - before < 64 * 2
    assert (eng.sampled(0) != 0).mean() > 0.9
    assert lib().rsd_debug_fail_iteration(eng.ctx, 3) == 0
    with pytest.raises(RsdError) as e:
        eng.step(0.0)
    assert e.value.code == -5
    assert (eng.sampled(0)[:, 1:] == 0).all()
    with pytest.raises(RsdError) as e:
        eng.step(0.0)
    assert e.value.code == -2
    eng.close()


@pytest.mark.parametrize("temperature", [0.0, 0.2, 0.7])
def test_speculative_rounds_that_sample_in_the_head(temperature):
    """From 65536 ids on proposals and the pass that verifies them sample in the head's epilogue, unless the target's logits are kept: the same tokens."""
    from paper_2501_19324_b200 import Engine, Model, RSD_DEBUG_KEEP_LOGITS
    sh = ri.ModelShape(2, 256, 2, 1, 128, 704, 65540)
    heads = (ri.HEAD_LM, ri.HEAD_REWARD_SIGMOID, ri.HEAD_LM)
    models = [Model(sh, ri.gpu_model_tensors(sh, slot, 0, True, hk), hk) for slot, hk in enumerate(heads)]
    prompts = ri.prompts(9, 6, 5, 40, sh.vocab)
    got = []
    for flags in (0, RSD_DEBUG_KEEP_LOGITS):
        eng = Engine(*models, max_batch=6, max_seq_tokens=100, max_step_tokens=12, max_steps=4, step_end_id=1, step_end_mod=20, temperature=temperature,
                     seed=2, sd_tokens=4, debug_flags=flags)
        eng.prefill(*prompts)
        steps = [eng.step(delta) for delta in (2.0, 0.0, 2.0)]
        got.append(([r["step_tokens"].tolist() for r in steps], eng.counters()))
        eng.close()
    assert got[0] == got[1]
    assert got[0][1]["sd_rounds"] > 0


def test_a_phase_without_rows_does_not_wait_for_the_stream():
    """No row has room for a step: the call returns although another thread keeps the caller's stream busy (for three seconds
    at most), since the phase says itself that it has nothing to decode."""
    import threading
    import time
    import torch
    prompts = ri.prompts(1, 3, 40, 40, MINI[0].vocab)
    eng = _engine(prompts, max_seq_tokens=64, max_step_tokens=32, max_steps=3, step_end_id=-1, temperature=0.0)
    assert not eng.step(0.0)["live"].any()
    stream, stop = torch.cuda.Stream(), threading.Event()

    def feed():
        end = time.monotonic() + 3.0
        with torch.cuda.stream(stream):
            pending = []
            while time.monotonic() < end and not stop.is_set():
                torch.cuda._sleep(2000000)               # about a millisecond
                pending.append(torch.cuda.Event())
                pending[-1].record()
                if len(pending) > 8:
                    pending.pop(0).synchronize()
    t = threading.Thread(target=feed)
    t.start()
    time.sleep(0.2)
    t0 = time.monotonic()
    with torch.cuda.stream(stream):
        out = eng.step(0.0)
    took = time.monotonic() - t0
    stop.set()
    t.join()
    torch.cuda.synchronize()
    assert not out["live"].any() and (out["step_len"] == 0).all()
    assert took < 1.5, took
    eng.close()


_BLOCKING = """
import ctypes, os, sys, time
sys.path[:0] = [{root!r}, os.path.join({root!r}, "tests")]
cuda = ctypes.CDLL("libcuda.so.1")
assert cuda.cuInit(0) == 0
if {blocking}:
    assert cuda.cuDevicePrimaryCtxSetFlags(0, 4) == 0            # CU_CTX_SCHED_BLOCKING_SYNC, this process only
import rsd_inputs as ri
from test_gpu_loop import MINI, _engine
eng = _engine(ri.prompts(1, 32, 40, 60, MINI[0].vocab), max_seq_tokens=600, max_step_tokens=120, max_steps=5, step_end_id=-1, temperature=0.7)
eng.step(0.0)
cpu, wall = time.thread_time(), time.perf_counter()
for _ in range(2):
    eng.step(0.0)
print("SHARE", (time.thread_time() - cpu) / (time.perf_counter() - wall))
"""


def test_a_blocking_process_sleeps_through_a_decode_phase():
    """A process that asked for blocking synchronisation has its thread asleep for much of a step; by default it polls."""
    import os
    import subprocess
    import sys
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    share = {}
    for blocking in (True, False):
        r = subprocess.run([sys.executable, "-c", _BLOCKING.format(root=root, blocking=blocking)], capture_output=True, text=True, timeout=240)
        assert r.returncode == 0, r.stderr[-2000:]
        share[blocking] = float(r.stdout.split("SHARE")[1])
    assert share[True] < 0.7 and share[True] < share[False], share


@pytest.mark.parametrize("C", [160, 170, 171, 690, 1500])        # 12 300 bytes each: below and above the line, less and more than the staging
def test_kept_logits_into_pageable_and_page_locked_memory(C):
    """The same bytes whichever way they come."""
    import torch
    from dataclasses import replace
    from paper_2501_19324_b200 import Engine, Model, lib, RSD_DEBUG_KEEP_LOGITS
    sh = [replace(s, vocab=1025) for s in TINY]
    models = [Model(s, ri.gpu_model_tensors(s, slot, 0, False, kind), kind) for slot, (s, kind) in enumerate(zip(sh, (ri.HEAD_LM, ri.HEAD_REWARD_SIGMOID, ri.HEAD_LM)))]
    eng = Engine(*models, max_batch=3, max_seq_tokens=C + 16, max_step_tokens=C, max_steps=1, step_end_id=3, debug_flags=RSD_DEBUG_KEEP_LOGITS)
    eng.prefill(*ri.prompts(1, 3, 5, 9, 1025))
    torch.manual_seed(C)
    eng._ws.random_(0, 256)                                            # the logits among them; nothing runs on it any more
    torch.cuda.synchronize()
    for which in (0, 2):
        locked = torch.empty(3, C, 1025, pin_memory=True)
        assert lib().rsd_debug_get_logits(eng.ctx, which, locked.data_ptr()) == 0
        got = eng.logits(which)
        assert got.shape == (3, C, 1025) and got.tobytes() == locked.numpy().tobytes()
    eng.close()
