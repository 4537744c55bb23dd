"""Each CUDA kernel against the oracle's function for the same operation, through the C ABI."""
import numpy as np
import pytest
import torch

import oracle
import rsd_inputs as ri
from paper_2501_19324_b200 import binding as rb

pytestmark = pytest.mark.gpu


def dev(a, dtype=None):
    t = torch.from_numpy(np.ascontiguousarray(a)).cuda()
    return t.to(dtype) if dtype is not None else t


def test_input_generators_agree_bit_for_bit():
    sh = ri.SHAPES["tiny_draft"]
    for bf16 in (False, True):
        g = ri.gpu_model_tensors(sh, 1, 3, bf16, ri.HEAD_REWARD_SIGMOID)
        c = ri.cpu_model_weights(sh, 1, 3, bf16, ri.HEAD_REWARD_SIGMOID)
        assert np.array_equal(g["tok_embed"].float().cpu().numpy(), c["tok_embed"])
        assert np.array_equal(g["head"].float().cpu().numpy(), c["head"])
        l = c["layers"][1]
        assert np.array_equal(g["wqkv"][1].float().cpu().numpy(), np.concatenate([l["wq"], l["wk"], l["wv"]]))
        assert np.array_equal(g["wgu"][1].float().cpu().numpy(), np.concatenate([l["wgate"], l["wup"]]))
        assert np.array_equal(g["wo"][1].float().cpu().numpy(), l["wo"])
        assert np.array_equal(g["wdown"][1].float().cpu().numpy(), l["wdown"])
        for k in ("norm1", "norm2"):
            assert np.array_equal(g[k][1].float().cpu().numpy(), l[k]) and np.abs(l[k] - 1).max() > 0.1
        assert np.array_equal(g["final_norm"].float().cpu().numpy(), c["final_norm"])


def philox_numpy(ctr, key):
    """Philox4x32-10 over an array of counters [n, 4] (uint32), written out with numpy integer arithmetic: ten rounds of
    two 32 x 32 -> 64-bit products whose halves are mixed with the other words and the key, the key advancing by the
    two Weyl constants.  A third statement of the algorithm beside the oracle's and the kernel's; the test checks it
    against the oracle before using it on every counter."""
    c = [ctr[:, i].astype(np.uint64) for i in range(4)]
    k0, k1 = np.uint64(key[0]), np.uint64(key[1])
    mask = np.uint64(0xFFFFFFFF)
    for _ in range(10):
        p0 = np.uint64(0xD2511F53) * c[0]
        p1 = np.uint64(0xCD9E8D57) * c[2]
        c = [(p1 >> np.uint64(32)) ^ c[1] ^ k0, p1 & mask, (p0 >> np.uint64(32)) ^ c[3] ^ k1, p0 & mask]
        k0 = (k0 + np.uint64(0x9E3779B9)) & mask
        k1 = (k1 + np.uint64(0xBB67AE85)) & mask
    return np.stack(c, axis=1).astype(np.uint32)


def test_philox_matches_oracle_on_many_counters():
    """2^20 random counters (plus all-zero and all-one words): every block of the kernel against the numpy
    restatement, which itself is checked against the oracle's C implementation on 512 of them."""
    rng = np.random.default_rng(0)
    n = 1 << 20
    ctr = rng.integers(0, 2 ** 32, size=(n, 4), dtype=np.uint64).astype(np.uint32)
    ctr[0] = 0
    ctr[1] = 0xFFFFFFFF
    key = np.array([0x12345678, 0x9ABCDEF0], dtype=np.uint32)
    want = philox_numpy(ctr, key)
    for i in list(range(64)) + list(rng.integers(0, n, size=448)):
        assert np.array_equal(want[i], oracle.philox4x32_10(ctr[i], key))
    got = rb.k_philox(dev(ctr.view(np.int32)), dev(key.view(np.int32))).cpu().numpy().view(np.uint32)
    assert np.array_equal(got, want)
    zero = rb.k_philox(dev(np.zeros((1, 4), np.int32)), dev(np.zeros(2, np.int32))).cpu().numpy().view(np.uint32)
    assert [hex(v) for v in zero[0]] == ["0x6627e8d5", "0xe169c58d", "0xbc57ac4c", "0x9b00dbd8"]


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("M,N,K", [(1, 1024, 256), (4, 688 * 2, 256), (7, 256, 688), (33, 1000, 512), (130, 257, 1024),
                                   (4, 40, 64), (5, 40, 64), (5, 512, 1376), (9, 2752, 512)])
def test_gemm_simt(M, N, K, bf16):
    rng = np.random.default_rng(M * 1000 + N)
    W = ri.cpu_tensor(1, 77, N, K, bf16)
    x = rng.normal(size=(M, K)).astype(np.float32)
    dt = torch.bfloat16 if bf16 else torch.float32
    xd = dev(x, dt)
    want = oracle.matmul(W, xd.float().cpu().numpy())
    y0 = rng.normal(size=(M, N)).astype(np.float32)
    got = rb.k_gemm(dev(W, dt), xd, impl=1).cpu().numpy()
    np.testing.assert_allclose(got, want, rtol=0, atol=2e-5 * np.sqrt(K))
    acc = rb.k_gemm(dev(W, dt), xd, y=dev(y0), accumulate=True, impl=1).cpu().numpy()
    np.testing.assert_allclose(acc, want + y0, rtol=0, atol=2e-5 * np.sqrt(K))


@pytest.mark.parametrize("M,N,K", [(17, 1928, 4), (33, 1000, 36), (97, 341, 688), (128, 256, 1376), (300, 130, 100),
                                   (17, 2412, 4), (41, 1000, 36), (121, 341, 688), (160, 257, 1376), (310, 130, 100)])
def test_gemm_fp32_of_many_rows(M, N, K):
    """The tiled fp32 product: less than a stage of K and many, ragged rows, columns and K; the bound of the test above."""
    test_gemm_simt(M, N, K, False)


def _fma32(a, b, c):
    return (a.astype(np.float64) * b.astype(np.float64) + c).astype(np.float32)


def _gemv_order(x, W, ks):
    """x W^T in fp32 in the order of the product of few rows: ks warps of 32 lanes, four values of K at a time, a tree over the lanes."""
    M, K, N, total = x.shape[0], x.shape[1], W.shape[0], np.float32(0)
    for split in range(ks):
        lanes = np.zeros((32, M, N), np.float32)
        for lane in range(32):
            for v in range(split * 32 + lane, K // 4, ks * 32):
                for k in range(4 * v, 4 * v + 4):
                    lanes[lane] = _fma32(x[:, k, None], W[None, :, k], lanes[lane])
        for o in (16, 8, 4, 2, 1):
            lanes = lanes[:o] + lanes[o:2 * o]
        total = total + lanes[0]
    return total


@pytest.mark.parametrize("M,N,K,ks", [(96, 512, 256, 1), (17, 2752, 512, 2), (96, 512, 1376, 4), (96, 512, 4096, 8)])
def test_gemm_fp32_of_many_rows_rounds_no_more(M, N, K, ks):
    """The tiled fp32 product's error against fp64 is no larger than that of the product of few rows at the K splits that it would take
    here.  Relative errors of 47k to 49k sums: their spread is 1 / sqrt(2 * 47k) = 0.33 %, of two of them 0.46 %; 1 % is allowed."""
    rng = np.random.default_rng(M + K)
    x = rng.standard_normal((M, K)).astype(np.float32)
    W = (0.05 * rng.standard_normal((N, K))).astype(np.float32)
    exact = x.astype(np.float64) @ W.T.astype(np.float64)
    got = rb.k_gemm(dev(W), dev(x), impl=1).cpu().numpy()
    assert np.linalg.norm(got - exact) <= 1.01 * np.linalg.norm(_gemv_order(x, W, ks) - exact)


@pytest.mark.parametrize("M,N,K", [(16, 128, 64), (5, 256, 512), (17, 1536, 1536), (32, 2048, 1536), (33, 1000, 520),
                                   (64, 1536, 8960), (100, 384, 1408), (128, 640, 768), (129, 256, 2048),
                                   (300, 4096, 512), (1000, 1280, 768), (8, 17920, 1536), (200, 384, 520), (2500, 1024, 192)])
def test_gemm_tcgen05(M, N, K):
    """Tensor-core path: ragged M, N not a multiple of the 128-row tile, K not a multiple of 64,
    split-K with the last-arriver reduction, several x tiles (more than 128 rows with a split operand take the
    persistent kernel: several tiles per CTA, more row tiles than one group of eight), accumulate into y."""
    rng = np.random.default_rng(M * 7 + N)
    W = ri.cpu_tensor(2, 5, N, K, True)
    x = rng.normal(size=(M, K)).astype(np.float32)
    xd = dev(x, torch.bfloat16)
    want = oracle.matmul(W, xd.float().cpu().numpy())
    Wd = dev(W, torch.bfloat16)
    got = rb.k_gemm(Wd, xd, impl=2).cpu().numpy()
    tol = 3e-5 * np.sqrt(K)
    np.testing.assert_allclose(got, want, rtol=0, atol=tol)
    y0 = rng.normal(size=(M, N)).astype(np.float32)
    acc = rb.k_gemm(Wd, xd, y=dev(y0), accumulate=True, impl=2).cpu().numpy()
    np.testing.assert_allclose(acc, want + y0, rtol=0, atol=tol)
    again = rb.k_gemm(Wd, xd, impl=2).cpu().numpy()
    assert np.array_equal(again, got)          # deterministic, whatever order the split CTAs finish in
    # split-precision activations: x = hi + lo, both bf16, both multiplied on the tensor cores
    xf = dev(x)
    hi = xf.to(torch.bfloat16)
    lo = (xf - hi.float()).to(torch.bfloat16)
    want2 = oracle.matmul(W, (hi.float() + lo.float()).cpu().numpy())
    got2 = rb.k_gemm(Wd, hi, impl=2, x_lo=lo).cpu().numpy()
    np.testing.assert_allclose(got2, want2, rtol=0, atol=tol)
    assert np.abs(want2 - oracle.matmul(W, x)).max() < 1e-3 * np.sqrt(K) * 0.02 + 1e-4   # hi + lo ~ x
    got3 = rb.k_gemm(Wd, hi, impl=1, x_lo=lo).cpu().numpy()                    # SIMT path, same operands
    np.testing.assert_allclose(got3, want2, rtol=0, atol=tol)


def test_rmsnorm_rope_swiglu():
    rng = np.random.default_rng(1)
    x = rng.normal(size=(5, 1536)).astype(np.float32) * 3
    g = (1 + 0.1 * rng.normal(size=1536)).astype(np.float32)
    got = rb.k_rmsnorm(dev(x), dev(g), 1e-6).cpu().numpy()
    want = np.stack([oracle.rmsnorm(x[i], g, 1e-6) for i in range(5)])
    np.testing.assert_allclose(got, want, rtol=0, atol=2e-6 * np.abs(want).max())
    got16 = rb.k_rmsnorm(dev(x), dev(g, torch.bfloat16), 1e-6).float().cpu().numpy()
    g16 = dev(g, torch.bfloat16).float().cpu().numpy()
    want16 = np.stack([oracle.rmsnorm(x[i], g16, 1e-6) for i in range(5)])
    np.testing.assert_allclose(got16, want16, rtol=2 ** -8, atol=0)

    for hd in (64, 128):
        v = rng.normal(size=(6, 3, hd)).astype(np.float32)
        pos = np.array([0, 1, 17, 255, 4095, 16383], dtype=np.int32)
        got = rb.k_rope(dev(v.copy()), dev(pos), 1e4).cpu().numpy()
        want = np.stack([[oracle.rope(v[t, h], pos[t], 1e4) for h in range(3)] for t in range(6)])
        np.testing.assert_allclose(got, want, rtol=0, atol=1e-6)

    gu = rng.normal(size=(4, 2 * 688)).astype(np.float32) * 2
    got = rb.k_swiglu(dev(gu), torch.float32).cpu().numpy()
    a, b = gu[:, :688].astype(np.float64), gu[:, 688:].astype(np.float64)
    np.testing.assert_allclose(got, a / (1 + np.exp(-a)) * b, rtol=1e-6, atol=1e-6)


@pytest.mark.parametrize("M,N,K", [(5, 256, 512), (40, 384, 1408), (100, 384, 1408), (128, 640, 768), (300, 384, 512)])
def test_gemm_buffers_may_start_anywhere(M, N, K):
    """Result at a 4-byte and scratch at an 8-byte boundary, with a K split (up to 128 rows) and without: the results of aligned
    buffers, added to y or not."""
    rng = np.random.default_rng(M)
    W = dev(ri.cpu_tensor(2, 5, N, K, True), torch.bfloat16)
    x = dev(rng.normal(size=(M, K)).astype(np.float32))
    hi = x.to(torch.bfloat16)
    lo = (x - hi.float()).to(torch.bfloat16)
    y0 = dev(rng.normal(size=(M, N)).astype(np.float32))
    nbytes = rb.lib().rsd_k_gemm_scratch_bytes(M, N, K)
    for accumulate in (0, 1):
        want = rb.k_gemm(W, hi, y=y0.clone(), accumulate=bool(accumulate), impl=2, x_lo=lo)
        y = torch.full((M * N + 4,), np.nan, device="cuda")
        y[1:M * N + 1] = y0.view(-1)
        scratch = torch.zeros(nbytes + 16, dtype=torch.uint8, device="cuda")
        assert rb.lib().rsd_k_gemm(W.data_ptr(), hi.data_ptr(), lo.data_ptr(), y.data_ptr() + 4, M, N, K, 1, accumulate, 2, scratch.data_ptr() + 8,
                                   nbytes, torch.cuda.current_stream().cuda_stream) == 0
        assert torch.equal(y[1:M * N + 1].view(M, N), want)
        assert bool(y[[0, -3, -2, -1]].isnan().all())


@pytest.mark.parametrize("d", [4, 252, 256, 260, 512, 516, 1024, 1028, 2048, 2052, 4096, 4100, 8192, 8196, 12288])
def test_rmsnorm_widths(d):
    """Both sides of every width at which the block or the vectors a thread keeps change, rows that are read again, and an output
    that starts off a 16-byte boundary.  A thread adds at most 24 squares, warps and block ten partial sums: 34 roundings of the
    sum, half of that in the root, and five more in root, quotient and products: 22 * 2^-24."""
    rng = np.random.default_rng(d)
    T = 3
    x = (rng.normal(size=(T, d)) * 3).astype(np.float32)
    g = (1 + 0.1 * rng.normal(size=d)).astype(np.float32)
    xd = x.astype(np.float64)
    root = np.sqrt((xd * xd).mean(axis=1, keepdims=True) + 1e-6)
    np.testing.assert_allclose(rb.k_rmsnorm(dev(x), dev(g), 1e-6).cpu().numpy(), xd * g / root, rtol=22 * 2.0 ** -24, atol=0)
    g16 = dev(g, torch.bfloat16)
    want16 = xd * g16.double().cpu().numpy() / root
    np.testing.assert_allclose(rb.k_rmsnorm(dev(x), g16, 1e-6).float().cpu().numpy(), want16, rtol=2 ** -8, atol=0)
    x_d, off = dev(x), torch.zeros(T * d + 8, dtype=torch.bfloat16, device="cuda")
    assert rb.lib().rsd_k_rmsnorm(x_d.data_ptr(), g16.data_ptr(), off.data_ptr() + 2, T, d, 1e-6, 1, torch.cuda.current_stream().cuda_stream) == 0
    np.testing.assert_allclose(off[1:T * d + 1].view(T, d).float().cpu().numpy(), want16, rtol=2 ** -8, atol=0)


@pytest.mark.parametrize("lo,hi", [(-1e-30, 1e-30), (-1.0, 1.0), (-30.0, 30.0), (-86.9, -80.0), (-88.7, -87.0), (-120.0, -87.0), (80.0, 1e4)])
def test_swiglu_over_its_range(lo, hi):
    """The exponential is good to 2 ulp, sum, quotient and product to half an ulp each: 3.5 ulp = 3.5 * 2^-23, plus an ulp for the
    step to the next binade.  Below -88.72 the exponential overflows and the result is zero: 2.7e-37 at most is lost, times up
    (|up| < 5 here)."""
    rng = np.random.default_rng(12)
    gu = np.concatenate([rng.uniform(lo, hi, (64, 512)), rng.normal(size=(64, 512))], axis=1).astype(np.float32)
    got = rb.k_swiglu(dev(gu), torch.float32).cpu().numpy()
    a, b = gu[:, :512].astype(np.float64), gu[:, 512:].astype(np.float64)
    np.testing.assert_allclose(got, a / (1 + np.exp(-a)) * b, rtol=4.5 * 2.0 ** -23, atol=5 * 2.7e-37 if lo < -88.72 else 2.0 ** -148)


def test_swiglu_is_the_division():
    """Every 61st float as the gate (all binades, both signs, infinities and NaNs among them) against gate / (1 + exp(-gate)) with
    CUDA's own division: the same value; where gate or result is subnormal, within a subnormal step."""
    gate = (torch.arange(0, 1 << 32, 61, device="cuda") - (1 << 31)).to(torch.int32).view(torch.float32)
    ends = torch.tensor([np.inf, -np.inf, np.nan, 3.4028235e38, -3.4028235e38, -1e30, -1e10, -104.0, -90.0, -88.8, -88.7, -87.1], device="cuda")
    gate = torch.cat([gate, ends])
    got = rb.k_swiglu(torch.cat([gate, torch.ones_like(gate)]).view(1, -1), torch.float32)[0]
    want = gate / (1 + torch.exp(-gate))
    assert torch.equal(torch.isnan(got), torch.isnan(want))
    tiny = (want.abs() < 2.0 ** -126) | (gate.abs() < 2.0 ** -124)
    same = (got == want) | torch.isnan(want) | (tiny & ((got.double() - want.double()).abs() <= 2.0 ** -148))
    assert bool(same.all()), (gate[~same][:8], got[~same][:8], want[~same][:8])


@pytest.mark.parametrize("temperature", [0.0, 0.7])
def test_sampling_matches_oracle(temperature):
    rng = np.random.default_rng(2)
    B, V, v_limit = 6, 5003, 4999
    logits = rng.normal(size=(B, V)).astype(np.float32)
    logits[0, 4] = logits[0, 9] = 50.0            # exact tie: lowest id wins when greedy
    logits[1, v_limit + 1] = 99.0                 # beyond the shared vocabulary: never chosen
    row = np.array([0, 1, 2, 3, -1, 7], dtype=np.int32)
    pos = np.array([5, 5, 9, 1000, 3, 70000], dtype=np.int32)
    got = rb.k_sample(dev(logits), v_limit, temperature, 1234, 2, dev(row), dev(pos)).cpu().numpy()
    for b in range(B):
        if row[b] < 0:
            continue
        want, margin = oracle.sample(logits[b].astype(np.float64), v_limit, temperature, 1234, 2, row[b], pos[b] + 1)
        if margin > 1e-4 or temperature == 0.0:
            assert got[b] == want, (b, got[b], want, margin)
    if temperature == 0.0:
        assert got[0] == 4


@pytest.mark.parametrize("v_limit,scale,shift", [(1, 1.0, 0.0), (4095, 1.0, 0.0), (4097, 4.0, 0.0), (16385, 30.0, 0.0), (65535, 0.8, 0.0),
                                                 (65537, 8.0, -50.0), (262145, 1.0, 2000.0)])
def test_sampling_shortcuts_keep_the_winner(v_limit, scale, shift):
    """Flat and peaked logits, a few large ones far above the rest, ids that the noise range rules out, large offsets (where
    one ulp of a score exceeds the shortcut's margin), infinite and NaN logits; one block per slot and many, full and
    ragged chunks, an odd row length (no 16-byte loads).  Against fp64 scores with the oracle's noise: the winner
    must be the oracle's unless its two best scores are within a few fp32 roundings of each other."""
    rng = np.random.default_rng(v_limit)
    B, V = 6, v_limit + 3
    logits = (rng.normal(size=(B, V)) * scale + shift).astype(np.float32)
    logits[1, rng.integers(0, v_limit, size=3)] += 25.0
    logits[2] = shift
    logits[3, :v_limit // 2] = -np.inf
    logits[4, rng.integers(0, v_limit, size=5)] = np.nan
    logits[4, v_limit - 1] = shift
    logits[:, v_limit:] = 1e9                                  # beyond the vocabulary limit: never chosen
    row, pos = np.arange(B, dtype=np.int32), np.arange(B, dtype=np.int32) * 37 + 5
    for temperature in (0.7, 0.0):
        got = rb.k_sample(dev(logits), v_limit, temperature, 77, 1, dev(row), dev(pos)).cpu().numpy()
        for b in range(B):
            fin = np.where(np.isnan(logits[b, :v_limit]), -np.inf, logits[b, :v_limit].astype(np.float64))
            want, margin = oracle.sample(np.concatenate([fin, np.full(3, -np.inf)]), v_limit, temperature, 77, 1, row[b], pos[b] + 1)
            if v_limit == 1 or temperature == 0.0 or margin > 4e-6 * (abs(shift) + 30 * scale) / 0.7:
                assert got[b] == want, (b, temperature, got[b], want, margin)


@pytest.mark.parametrize("v_limit,scale,shift", [(127, 1.0, 0.0), (1024, 8.0, 0.0), (4097, 4.0, 0.0), (16385, 30.0, 0.0), (65537, 8.0, -50.0), (151936, 1.0, 2000.0)])
def test_sampling_forms_agree(v_limit, scale, shift):
    """Few ids in all take exact noise at once, more than 1.5 million the shortcuts: a handful of rows alone and the same rows
    repeated until the call is beyond that line must give the same ids (both forms compare the same exact scores)."""
    rng = np.random.default_rng(v_limit + 1)
    B, V = 5, v_limit + 2
    logits = (rng.normal(size=(B, V)) * scale + shift).astype(np.float32)
    logits[1, rng.integers(0, v_limit, size=3)] += 25.0
    logits[2] = shift
    logits[3, :v_limit // 2] = -np.inf
    logits[4, rng.integers(0, v_limit, size=5)] = np.nan
    row, pos = np.arange(B, dtype=np.int32), np.arange(B, dtype=np.int32) * 41 + 3
    reps = 1500000 // (B * v_limit) + 1
    for temperature in (0.7, 0.0):
        few = rb.k_sample(dev(logits), v_limit, temperature, 91, 0, dev(row), dev(pos))
        many = rb.k_sample(dev(logits).repeat(reps, 1), v_limit, temperature, 91, 0, dev(row).repeat(reps), dev(pos).repeat(reps))
        assert B * v_limit <= 1500000 < reps * B * v_limit
        assert torch.equal(many.view(reps, B), few.expand(reps, B)), temperature


def test_gate_compaction_all_masks_and_large():
    """Brute force (a serial loop over the rows) against the ballot / prefix path: EVERY accept mask of 12 rows, one
    call per mask as the step loop calls it, and every mask of 16 rows laid end to end in one call of 2^20 rows."""
    B = 12
    n_masks = 1 << B
    bits = (np.arange(n_masks)[:, None] >> np.arange(B)[None, :]) & 1               # [mask, row]
    r = np.where(bits == 1, np.float32(0.9), np.float32(0.1)).astype(np.float32)
    live = np.tile(np.array([1 if b % 5 else 0 for b in range(B)], dtype=np.uint8), (n_masks, 1))
    r_d, live_d = dev(r), dev(live)
    acc_d = torch.zeros(n_masks, B, dtype=torch.uint8, device="cuda")
    rej_d = torch.full((n_masks, B), -1, dtype=torch.int32, device="cuda")
    n_d = torch.zeros(n_masks, dtype=torch.int32, device="cuda")
    scratch = torch.zeros(64, dtype=torch.uint8, device="cuda")
    stream = torch.cuda.current_stream().cuda_stream
    for m in range(n_masks):
        rc = rb.lib().rsd_k_gate_compact(r_d.data_ptr() + 4 * B * m, live_d.data_ptr() + B * m, 0.5, acc_d.data_ptr() + B * m,
                                         rej_d.data_ptr() + 4 * B * m, n_d.data_ptr() + 4 * m, B, scratch.data_ptr(), 64, stream)
        assert rc == 0
    acc, rej, n = acc_d.cpu().numpy(), rej_d.cpu().numpy(), n_d.cpu().numpy()
    for m in range(n_masks):
        want_rej = []
        for b in range(B):                                  # the serial definition
            if live[m, b] and not (r[m, b] >= np.float32(0.5)):
                want_rej.append(b)
        assert n[m] == len(want_rej), m
        assert rej[m, :len(want_rej)].tolist() == want_rej, m
        assert acc[m].tolist() == [int(live[m, b] and r[m, b] >= np.float32(0.5)) for b in range(B)], m
    # all 2^16 masks of 16 rows as consecutive segments of one call: the ascending global list, cut at the
    # segment boundaries, is every segment's own ascending list
    B = 16
    n_masks = 1 << B
    bits = (np.arange(n_masks)[:, None] >> np.arange(B)[None, :]) & 1
    r = np.where(bits == 1, np.float32(0.9), np.float32(0.1)).astype(np.float32).reshape(-1)
    live = np.tile(np.array([0 if b in (3, 11) else 1 for b in range(B)], dtype=np.uint8), n_masks)
    acc, rej, n = rb.k_gate_compact(dev(r), dev(live), 0.5)
    acc, rej, n = acc.cpu().numpy(), rej.cpu().numpy(), int(n.item())
    want = []
    for i in range(n_masks * B):
        if live[i] and not (r[i] >= np.float32(0.5)):
            want.append(i)
    assert n == len(want) and np.array_equal(rej[:n], np.array(want, dtype=np.int32))
    assert np.array_equal(acc, ((live == 1) & (r >= np.float32(0.5))).astype(np.uint8))
    seg = rej[:n] // B
    for m in (0, 1, 0x5A5A, 0xFFFF, 0x8001):
        want_rej = [b for b in range(B) if live[m * B + b] and not ((m >> b) & 1)]
        assert (rej[:n][seg == m] - m * B).tolist() == want_rej
    rng = np.random.default_rng(3)
    for B, p in [(1, 0.5), (1023, 0.3), (1024, 0.9), (1025, 0.1), (70001, 0.7), (1 << 20, 0.5)]:
        r = rng.random(B).astype(np.float32)
        live = (rng.random(B) < 0.95).astype(np.uint8)
        delta = np.float32(1 - p)
        acc, rej, n = rb.k_gate_compact(dev(r), dev(live), float(delta))
        want = np.nonzero((live == 1) & ~(r >= delta))[0]
        assert int(n.item()) == len(want)
        assert np.array_equal(rej.cpu().numpy()[:len(want)], want)
        assert np.array_equal(acc.cpu().numpy(), ((live == 1) & (r >= delta)).astype(np.uint8))
    # r == delta accepts; NaN rejects
    r = np.array([0.7, np.nan, np.nextafter(np.float32(0.7), np.float32(0))], dtype=np.float32)
    acc, rej, n = rb.k_gate_compact(dev(r), dev(np.ones(3, np.uint8)), 0.7)
    assert acc.cpu().numpy().tolist() == [1, 0, 0] and rej.cpu().numpy()[:2].tolist() == [1, 2]


def paged_kv(rng, B, KV, hd, ctx, dtype, max_pages, ext=False):
    """Random K/V per row scattered over randomly permuted pages; returns pool, table, dense K, V.
    ext: pages carry two more blocks with the low halves of keys and values (x = fp16 hi + fp16 lo)."""
    n_pages_row = [(c + 15) // 16 for c in ctx]
    total = sum(n_pages_row)
    perm = rng.permutation(total + 5)
    # page = keys [KV][16][hd] followed by values transposed [KV][hd][16]; unused slots hold NaN
    pool = np.full((total + 5, 4 if ext else 2, KV * 16 * hd), np.nan, dtype=np.float32)
    table = np.zeros((B, max_pages), dtype=np.int32)
    Ks, Vs = [], []
    nxt = 0
    for b in range(B):
        K = rng.normal(size=(ctx[b], KV, hd)).astype(np.float32)
        V = rng.normal(size=(ctx[b], KV, hd)).astype(np.float32)
        for i in range(n_pages_row[b]):
            pg = perm[nxt]; nxt += 1
            table[b, i] = pg
            n = min(16, ctx[b] - 16 * i)
            kk = pool[pg, 0].reshape(KV, 16, hd)
            vv = pool[pg, 1].reshape(KV, hd, 16)
            kblk = K[16 * i:16 * i + n].transpose(1, 0, 2)
            if ext:
                khi = kblk.astype(np.float16).astype(np.float32)
                kk[:, :n] = khi
                pool[pg, 2].reshape(KV, 16, hd)[:, :n] = kblk - khi
            else:
                kk[:, :n] = kblk
            vblk = V[16 * i:16 * i + n].transpose(1, 2, 0)
            if ext:
                vhi = vblk.astype(np.float16).astype(np.float32)
                vv[:, :, :n] = vhi
                pool[pg, 3].reshape(KV, hd, 16)[:, :, :n] = vblk - vhi
            else:
                vv[:, :, :n] = vblk
        Ks.append(K); Vs.append(V)
    pool_d = dev(pool, dtype)
    pool_back = pool_d.float().cpu().numpy()
    for b in range(B):       # the oracle sees the values as stored (bf16-rounded when 16-bit)
        for i in range(n_pages_row[b]):
            n = min(16, ctx[b] - 16 * i)
            Ks[b][16 * i:16 * i + n] = pool_back[table[b, i], 0].reshape(KV, 16, hd)[:, :n].transpose(1, 0, 2)
            Vs[b][16 * i:16 * i + n] = pool_back[table[b, i], 1].reshape(KV, hd, 16)[:, :, :n].transpose(2, 0, 1)
            if ext:
                Ks[b][16 * i:16 * i + n] += pool_back[table[b, i], 2].reshape(KV, 16, hd)[:, :n].transpose(1, 0, 2)
                Vs[b][16 * i:16 * i + n] += pool_back[table[b, i], 3].reshape(KV, hd, 16)[:, :, :n].transpose(2, 0, 1)
    return pool_d, dev(table), Ks, Vs


@pytest.mark.parametrize("dtype,hd,H,KV", [(torch.float32, 64, 4, 2), (torch.bfloat16, 128, 12, 2),
                                          (torch.bfloat16, 128, 28, 4), (torch.bfloat16, 128, 8, 1),
                                          (torch.bfloat16, 64, 6, 2), (torch.bfloat16, 128, 16, 1),
                                          (torch.bfloat16, 128, 64, 8), (torch.float16, 128, 12, 2),
                                          (torch.float16, 64, 4, 2), (torch.float16, 128, 28, 4)])
def test_decode_attention_against_definition(dtype, hd, H, KV):
    rng = np.random.default_rng(4)
    ctx = [1, 15, 16, 17, 33, 250, 1031, 2049]
    B = len(ctx)
    max_pages = 130
    # fp32 caches: fp32 arithmetic.  bf16 caches: the query and the softmax weights are rounded to
    # bf16 for the tensor-core products (relative 2^-9 each) on values of order one
    tol = {torch.float32: 2e-5, torch.bfloat16: 1.5e-2, torch.float16: 2e-3}[dtype]
    pool, table, Ks, Vs = paged_kv(rng, B, KV, hd, ctx, dtype, max_pages)
    q = rng.normal(size=(B, H, hd)).astype(np.float32)
    got = rb.k_attn_decode(dev(q), pool, table, dev(np.array(ctx, np.int32)), KV).cpu().numpy()
    for b in range(B):
        for h in range(H):
            g = h // (H // KV)
            s = Ks[b][:, g].astype(np.float64) @ q[b, h].astype(np.float64) / np.sqrt(hd)
            p = np.exp(s - s.max()); p /= p.sum()
            want = p @ Vs[b][:, g].astype(np.float64)
            np.testing.assert_allclose(got[b, h], want, rtol=0, atol=tol)


@pytest.mark.parametrize("hd,H,KV", [(128, 28, 4), (64, 4, 2)])
@pytest.mark.parametrize("B,max_pages", [(1, 15), (2, 16), (1, 200), (70, 24), (3, 520)])
def test_decode_attention_at_the_edges_of_the_split_rule(hd, H, KV, B, max_pages):
    """One split, two, eight in a cluster, more than a cluster holds (merge launch), one per row, and splits of more pages
    than the ring holds; the longest row fills its page table, others end at a page's edge, in its first token, or after
    one token.  Tolerance: the query and the softmax weights are rounded to fp16 (2^-11 relative each)."""
    rng = np.random.default_rng(B * 1000 + max_pages)
    ctx = [max_pages * 16] + [int(c) for c in rng.integers(1, max_pages * 4, size=B - 1)]
    if B > 2:
        ctx[1], ctx[2] = 1, 33
    pool, table, Ks, Vs = paged_kv(rng, B, KV, hd, ctx, torch.float16, max_pages)
    q = rng.normal(size=(B, H, hd)).astype(np.float32)
    got = rb.k_attn_decode(dev(q), pool, table, dev(np.array(ctx, np.int32)), KV).cpu().numpy()
    for b in range(B):
        for h in range(0, H, max(1, H // 4)):
            g = h // (H // KV)
            s = Ks[b][:, g].astype(np.float64) @ q[b, h].astype(np.float64) / np.sqrt(hd)
            p = np.exp(s - s.max()); p /= p.sum()
            np.testing.assert_allclose(got[b, h], p @ Vs[b][:, g].astype(np.float64), rtol=0, atol=2e-3)


@pytest.mark.parametrize("hd,H,KV,B,max_pages", [(128, 28, 4, 1, 5), (128, 28, 4, 1, 6), (128, 28, 4, 2, 9), (64, 4, 2, 4, 31), (128, 12, 2, 5, 12), (128, 12, 2, 5, 13),
                                                 (128, 28, 4, 8, 14), (128, 28, 4, 9, 15), (128, 12, 2, 1, 192), (128, 12, 2, 1, 193)])
def test_decode_attention_of_few_rows_in_short_splits(hd, H, KV, B, max_pages):
    """Either side of the lines between one split, a page a split, three pages a split and more splits than a cluster holds."""
    test_decode_attention_at_the_edges_of_the_split_rule(hd, H, KV, B, max_pages)


@pytest.mark.parametrize("dtype,hd,H,KV", [(torch.float32, 64, 4, 2), (torch.float32, 128, 3, 3), (torch.float16, 128, 18, 2),
                                          (torch.bfloat16, 64, 9, 1)])
def test_generic_attention_at_the_edges_of_a_round_of_warps(dtype, hd, H, KV):
    """fp32 caches and groups wider than eight heads: contexts of fewer pages than the block has warps, exactly one page
    a warp (128 tokens with eight warps, 256 with sixteen), one token more, and a second round; the unused slots hold
    NaN.  fp32 arithmetic on the stored values: about 300 products and sums of order one, each rounded to 2^-24."""
    rng = np.random.default_rng(12)
    ctx = [1, 112, 127, 128, 129, 145, 256, 257]
    pool, table, Ks, Vs = paged_kv(rng, len(ctx), KV, hd, ctx, dtype, 20)
    q = rng.normal(size=(len(ctx), H, hd)).astype(np.float32)
    got = rb.k_attn_decode(dev(q), pool, table, dev(np.array(ctx, np.int32)), KV).cpu().numpy()
    for b in range(len(ctx)):
        for h in range(H):
            g = h // (H // KV)
            s = Ks[b][:, g].astype(np.float64) @ q[b, h].astype(np.float64) / np.sqrt(hd)
            p = np.exp(s - s.max()); p /= p.sum()
            np.testing.assert_allclose(got[b, h], p @ Vs[b][:, g].astype(np.float64), rtol=0, atol=2e-5)


@pytest.mark.parametrize("dtype,hd,H,KV", [(torch.float16, 128, 12, 2), (torch.float16, 128, 28, 4), (torch.float16, 64, 4, 2),
                                          (torch.float32, 64, 4, 2), (torch.float16, 128, 64, 8), (torch.float16, 128, 8, 4),
                                          (torch.float16, 128, 3, 3), (torch.bfloat16, 128, 12, 2)])
def test_chunk_attention_against_definition(dtype, hd, H, KV):
    """Ragged chunks of several rows in one list: tiles that straddle rows, a chunk that starts in the
    middle of a page, long prefixes, one idle entry; every query against brute-force causal softmax."""
    rng = np.random.default_rng(8)
    ctx = [40, 1, 300, 17, 1031]                # cached positions per row after the chunk was written
    new = [40, 1, 37, 5, 70]                    # the last `new` positions of each row are the chunk
    B = len(ctx)
    max_pages = 70
    pool, table, Ks, Vs = paged_kv(rng, B, KV, hd, ctx, dtype, max_pages)
    rows, poss = [], []
    for b in range(B):
        for p in range(ctx[b] - new[b], ctx[b]):
            rows.append(b); poss.append(p)
    rows.insert(45, -1); poss.insert(45, 0)     # an idle entry in the middle of the list
    T = len(rows)
    q = rng.normal(size=(T, H, hd)).astype(np.float32)
    got = rb.k_attn_chunk(dev(q), pool, table, dev(np.array(rows, np.int32)), dev(np.array(poss, np.int32)), KV).cpu().numpy()
    tol = {torch.float32: 2e-5, torch.float16: 2e-3, torch.bfloat16: 1.5e-2}[dtype]
    for t in range(T):
        b, p = rows[t], poss[t]
        if b < 0:
            continue
        for h in range(0, H, max(1, H // 6)):
            g = h // (H // KV)
            s = Ks[b][:p + 1, g].astype(np.float64) @ q[t, h].astype(np.float64) / np.sqrt(hd)
            w = np.exp(s - s.max()); w /= w.sum()
            want = w @ Vs[b][:p + 1, g].astype(np.float64)
            np.testing.assert_allclose(got[t, h], want, rtol=0, atol=tol)


@pytest.mark.parametrize("H,KV", [(12, 2), (28, 4), (8, 1), (3, 3), (18, 3), (64, 8), (24, 24)])
def test_long_chunk_attention_one_pass(H, KV):
    """More than 1024 entries: rows of one token, rows that end inside a key tile, at its edge and one token on; tiles that
    straddle rows, an idle entry, prefixes of several key tiles; scores that rise along the context so that the reference
    maximum is raised again and again (keys scaled up with the position), and rows whose largest score comes first.  Against
    brute-force softmax; the query and the weights are rounded to fp16 (2^-11 relative each), outputs are of order one."""
    rng = np.random.default_rng(15)
    ctx = [1, 128, 129, 700, 511, 260]
    new = [1, 128, 100, 600, 250, 130]
    max_pages = 48
    pool, table, Ks, Vs = paged_kv(rng, len(ctx), KV, 128, ctx, torch.float16, max_pages)
    raw = pool.float().cpu().numpy()
    for b, grow in ((3, 1), (4, -1)):                  # scale the keys of row 3 up along the context, of row 4 down
        for i in range((ctx[b] + 15) // 16):
            f = 1 + (0.5 * i if grow > 0 else 0.5 * (31 - i))
            raw[table[b, i].item(), 0] *= np.float32(f)
    pool = torch.from_numpy(raw).cuda().to(torch.float16)
    back = pool.float().cpu().numpy()
    for b in (3, 4):
        for i in range((ctx[b] + 15) // 16):
            n = min(16, ctx[b] - 16 * i)
            Ks[b][16 * i:16 * i + n] = back[table[b, i].item(), 0].reshape(KV, 16, 128)[:, :n].transpose(1, 0, 2)
    rows, poss = [], []
    for b in range(len(ctx)):
        for p in range(ctx[b] - new[b], ctx[b]):
            rows.append(b); poss.append(p)
    rows.insert(45, -1); poss.insert(45, 0)
    T = len(rows)
    assert T > 1024
    q = rng.normal(size=(T, H, 128)).astype(np.float32)
    got = rb.k_attn_chunk(dev(q), pool, table, dev(np.array(rows, np.int32)), dev(np.array(poss, np.int32)), KV).cpu().numpy()
    assert np.isfinite(got[np.array(rows) >= 0]).all()
    # a score s enters as fp16(q) . K: it errs by |s| 2^-11 / sqrt(hd) or so, and the weights by as much in relative terms
    for t in list(range(0, T, 17)) + [44, 46, T - 1]:
        b, p = rows[t], poss[t]
        if b < 0:
            continue
        for h in range(0, H, max(1, H // 4)):
            g = h // (H // KV)
            qh = q[t, h].astype(np.float64)
            s = Ks[b][:p + 1, g].astype(np.float64) @ qh / np.sqrt(128)
            w = np.exp(s - s.max()); w /= w.sum()
            tol = 2e-3 + 2 ** -11 * np.abs(Ks[b][:p + 1, g]).max() * 4
            np.testing.assert_allclose(got[t, h], w @ Vs[b][:p + 1, g].astype(np.float64), rtol=0, atol=tol)


@pytest.mark.parametrize("H,KV", [(28, 4), (12, 2)])
def test_chunk_attention_long_prefix(H, KV):
    """Prefixes of more than a hundred pages (the page ids of a row are fetched in batches of 32, several batches a
    pass), a chunk that ends in the middle of a page, two rows in one tile; fp16 cache, head_dim 128."""
    rng = np.random.default_rng(21)
    hd = 128
    ctx = [2603, 531]
    new = [90, 70]
    B = len(ctx)
    max_pages = 170
    pool, table, Ks, Vs = paged_kv(rng, B, KV, hd, ctx, torch.float16, max_pages)
    rows, poss = [], []
    for b in range(B):
        for p in range(ctx[b] - new[b], ctx[b]):
            rows.append(b); poss.append(p)
    T = len(rows)
    q = rng.normal(size=(T, H, hd)).astype(np.float32)
    got = rb.k_attn_chunk(dev(q), pool, table, dev(np.array(rows, np.int32)), dev(np.array(poss, np.int32)), KV).cpu().numpy()
    assert np.isfinite(got).all()
    for t in range(0, T, 3):
        b, p = rows[t], poss[t]
        for h in range(0, H, max(1, H // 5)):
            g = h // (H // KV)
            s = Ks[b][:p + 1, g].astype(np.float64) @ q[t, h].astype(np.float64) / np.sqrt(hd)
            w = np.exp(s - s.max()); w /= w.sum()
            want = w @ Vs[b][:p + 1, g].astype(np.float64)
            np.testing.assert_allclose(got[t, h], want, rtol=0, atol=2e-3)


@pytest.mark.parametrize("ctx", [[5, 100, 33], [700, 400, 3], [9000]])
def test_decode_attention_buffers_may_start_anywhere(ctx):
    """One split, a cluster of splits, more splits than a cluster: output at a 4-byte and scratch at an 8-byte boundary give the
    results of aligned buffers."""
    rng = np.random.default_rng(31)
    H, KV, hd, B = 12, 2, 128, len(ctx)
    max_pages = (max(ctx) + 15) // 16
    pool, table, _, _ = paged_kv(rng, B, KV, hd, ctx, torch.float16, max_pages)
    q, lens = dev(rng.normal(size=(B, H, hd)).astype(np.float32)), dev(np.array(ctx, np.int32))
    want = rb.k_attn_decode(q, pool, table, lens, KV)
    nbytes = rb.lib().rsd_k_attn_decode_scratch_bytes(B, H, hd, max_pages * 16)
    out = torch.full((B * H * hd + 4,), np.nan, device="cuda")
    scratch = torch.empty(nbytes + 16, dtype=torch.uint8, device="cuda")
    assert rb.lib().rsd_k_attn_decode(q.data_ptr(), pool.data_ptr(), table.data_ptr(), lens.data_ptr(), out.data_ptr() + 4, B, H, KV, hd, max_pages,
                                      2, scratch.data_ptr() + 8, nbytes, torch.cuda.current_stream().cuda_stream) == 0
    assert torch.equal(out[1:B * H * hd + 1].view(B, H, hd), want)
    assert bool(out[[0, -3, -2, -1]].isnan().all())


@pytest.mark.parametrize("dtype,hd,H,KV", [(torch.float32, 64, 4, 2), (torch.float32, 128, 6, 3), (torch.float16, 64, 18, 1), (torch.bfloat16, 128, 16, 1)])
def test_generic_attention_pool_may_start_anywhere(dtype, hd, H, KV):
    """fp32 caches and groups of more than eight heads: a pool that starts one element off a 16-byte boundary."""
    rng = np.random.default_rng(32)
    ctx = [1, 16, 75, 300]
    pool, table, _, _ = paged_kv(rng, len(ctx), KV, hd, ctx, dtype, 20)
    q, lens = dev(rng.normal(size=(len(ctx), H, hd)).astype(np.float32)), dev(np.array(ctx, np.int32))
    want = rb.k_attn_decode(q, pool, table, lens, KV)
    moved = torch.empty(pool.numel() + 1, dtype=dtype, device="cuda")[1:].view(pool.shape)
    moved.copy_(pool)
    assert moved.data_ptr() % 16 == dtype.itemsize
    assert torch.equal(rb.k_attn_decode(q, moved, table, lens, KV), want)


@pytest.mark.parametrize("dtype,ext", [(torch.float16, False), (torch.bfloat16, False), (torch.float16, True)])
def test_tensor_core_attention_refuses_pools_off_a_boundary(dtype, ext):
    """These kernels copy 16 bytes at a time: a pool one element off is an argument error, before anything runs."""
    H, KV, hd = 8, 2, 64
    pool = torch.zeros(4 * KV * 16 * hd + 8, dtype=dtype, device="cuda")[1:]
    q = torch.zeros(1, H, hd, device="cuda")
    one = torch.ones(1, dtype=torch.int32, device="cuda")
    table = torch.zeros(1, 1, dtype=torch.int32, device="cuda")
    for call in (lambda: rb.k_attn_decode(q, pool, table, one, KV, ext=ext),
                 lambda: rb.k_attn_chunk(q, pool, table, torch.zeros_like(one), one, KV, ext=ext)):
        with pytest.raises(rb.RsdError) as e:
            call()
        assert e.value.code == -1


@pytest.mark.parametrize("hd,H,KV", [(128, 12, 2), (128, 64, 8), (64, 4, 2), (128, 16, 1)])
def test_extended_precision_attention(hd, H, KV):
    """fp16 cache with keys and values kept as hi + lo pairs, queries and softmax weights as hi + lo
    pairs: decode and chunk kernels alike agree with the fp64 definition to fp32 accuracy."""
    rng = np.random.default_rng(12)
    ctx = [1, 16, 33, 250, 1031]
    B = len(ctx)
    pool, table, Ks, Vs = paged_kv(rng, B, KV, hd, ctx, torch.float16, 70, ext=True)
    q = rng.normal(size=(B, H, hd)).astype(np.float32)
    got = rb.k_attn_decode(dev(q), pool, table, dev(np.array(ctx, np.int32)), KV, ext=True).cpu().numpy()
    rows = [b for b in range(B) for _ in range(min(ctx[b], 20))]
    poss = [p for b in range(B) for p in range(ctx[b] - min(ctx[b], 20), ctx[b])]
    qc = rng.normal(size=(len(rows), H, hd)).astype(np.float32)
    gotc = rb.k_attn_chunk(dev(qc), pool, table, dev(np.array(rows, np.int32)), dev(np.array(poss, np.int32)), KV, ext=True).cpu().numpy()

    def ref(b, p, qv, h):
        g = h // (H // KV)
        s = Ks[b][:p + 1, g].astype(np.float64) @ qv.astype(np.float64) / np.sqrt(hd)
        w = np.exp(s - s.max()); w /= w.sum()
        return w @ Vs[b][:p + 1, g].astype(np.float64)
    for b in range(B):
        for h in range(0, H, max(1, H // 4)):
            np.testing.assert_allclose(got[b, h], ref(b, ctx[b] - 1, q[b, h], h), rtol=0, atol=2e-5)
    for t in range(0, len(rows), 3):
        for h in range(0, H, max(1, H // 4)):
            np.testing.assert_allclose(gotc[t, h], ref(rows[t], poss[t], qc[t, h], h), rtol=0, atol=2e-5)


@pytest.mark.parametrize("M,N,K", [(129, 256, 64), (300, 1000, 520), (512, 1536, 1536), (2100, 640, 128), (4096, 2048, 1536)])
def test_dense_gemm_on_fp16_operands(M, N, K):
    """The dense form of the long passes (rsd_k_gemm impl 4): fp16 weights x one fp16 activation operand, more than
    128 rows, with and without adding into y; against the exact product of the fp16 values in fp64."""
    rng = np.random.default_rng(31)
    W = (rng.normal(size=(N, K)) * 0.05).astype(np.float16)
    x = rng.normal(size=(M, K)).astype(np.float16)
    want = x.astype(np.float64) @ W.astype(np.float64).T
    Wd, xd = torch.from_numpy(W).cuda(), torch.from_numpy(x).cuda()
    got = rb.k_gemm(Wd, xd, impl=4).cpu().numpy()
    tol = 2e-5 * np.sqrt(K) + 1e-6                      # fp32 accumulation of K products of order 0.05
    np.testing.assert_allclose(got, want, rtol=0, atol=tol)
    y0 = rng.normal(size=(M, N)).astype(np.float32)
    got2 = rb.k_gemm(Wd, xd, y=torch.from_numpy(y0.copy()).cuda(), accumulate=True, impl=4).cpu().numpy()
    np.testing.assert_allclose(got2, want + y0, rtol=0, atol=tol + 1e-6)
    with pytest.raises(rb.RsdError):
        rb.k_gemm(Wd, xd[:128].contiguous(), impl=4)    # the form is for more than 128 rows


@pytest.mark.parametrize("M", [1665, 2047, 3072, 3073])
def test_dense_gemm_that_adds_over_a_short_k(M):
    """Twelve weight tiles: up to 3072 rows make fewer 256-row tiles than SMs and are taken 128 rows at a time, one row more is not;
    fp32 sums of K products of order 0.05."""
    N, K = 1536, 136
    rng = np.random.default_rng(M)
    W = (rng.normal(size=(N, K)) * 0.05).astype(np.float16)
    x, y0 = rng.normal(size=(M, K)).astype(np.float16), rng.normal(size=(M, N)).astype(np.float32)
    got = rb.k_gemm(dev(W), dev(x), y=dev(y0.copy()), accumulate=True, impl=4).cpu().numpy()
    np.testing.assert_allclose(got, x.astype(np.float64) @ W.astype(np.float64).T + y0, rtol=0, atol=2e-5 * np.sqrt(K) + 2e-6)


@pytest.mark.parametrize("M,F,K", [(1, 64, 64), (5, 192, 512), (32, 1408, 512), (33, 128, 520), (70, 2048, 768),
                                   (129, 704, 1408), (300, 320, 256), (32, 8960, 1536), (200, 128, 520), (2100, 640, 128),
                                   (65, 9536, 192), (128, 9472, 520)])
def test_gate_up_gemm_with_swiglu_epilogue(M, F, K):
    """Gate/up projection with SwiGLU inside the GEMM epilogue (tile = 64 gate rows + the 64 matching up rows):
    against matmul + silu(g) * u written out in fp64.  Ragged M (all three tile heights and several x tiles), F of
    one to many tiles, K not a multiple of 64; the hi + lo output pair must carry the result to ~16 bits."""
    rng = np.random.default_rng(M * 13 + F)
    W = ri.cpu_tensor(3, 7, 2 * F, K, True) * 8.0          # pre-activations of order one, so silu is exercised
    W = dev(W, torch.bfloat16).float().cpu().numpy()
    x = rng.normal(size=(M, K)).astype(np.float32)
    xf = dev(x)
    hi = xf.to(torch.bfloat16)
    lo = (xf - hi.float()).to(torch.bfloat16)
    gu = oracle.matmul(W, (hi.float() + lo.float()).cpu().numpy()).astype(np.float64)
    g, u = gu[:, :F], gu[:, F:]
    want = g / (1.0 + np.exp(-g)) * u
    a_hi, a_lo = rb.k_gemm_gu(dev(W, torch.bfloat16), hi, lo)
    got = a_hi.float().cpu().numpy().astype(np.float64) + a_lo.float().cpu().numpy()
    scale = max(1.0, float(np.abs(want).max()))
    np.testing.assert_allclose(got, want, rtol=0, atol=(3e-5 * np.sqrt(K) + 2e-5) * scale)
    assert np.array_equal(a_hi.float().cpu().numpy(), torch.from_numpy(got.astype(np.float32)).to(torch.bfloat16).float().numpy()) or \
        np.abs(a_hi.float().cpu().numpy() - got).max() <= 2 ** -8 * scale
    again_hi, again_lo = rb.k_gemm_gu(dev(W, torch.bfloat16), hi, lo)
    assert torch.equal(again_hi, a_hi) and torch.equal(again_lo, a_lo)


@pytest.mark.parametrize("M,F,K", [(2, 1408, 512), (8, 192, 520), (9, 128, 768), (16, 18944, 256), (17, 64, 520)])
def test_gate_up_tiles_of_few_rows(M, F, K):
    """Tiles of 8, 16 and 32 rows at their edges: full, one row into the next, one or two CTAs per SM; the bound of the test above."""
    test_gate_up_gemm_with_swiglu_epilogue(M, F, K)


@pytest.mark.parametrize("M,N,K", [(65, 128, 64), (65, 1536, 8960), (128, 640, 520), (96, 18816, 128), (65, 18945, 192), (128, 19072, 520)])
def test_paired_gemm_of_65_to_128_rows(M, N, K):
    """The decode products of large batches: K split over the SMs (the smallest, a long K with many splits, a K tail), a
    weight matrix of 147 tiles (one wave) and of more than 148 (persistent kernel, ragged last tile).  fp32 sums of K
    products of N(0, 1) activations and N(0, 0.02) weights: about 2^-24 * K * 0.02, bounded as in the tests above."""
    rng = np.random.default_rng(M * 11 + N)
    W = ri.cpu_tensor(2, 9, N, K, True)
    xf = dev(rng.normal(size=(M, K)).astype(np.float32))
    hi = xf.to(torch.bfloat16)
    lo = (xf - hi.float()).to(torch.bfloat16)
    want = oracle.matmul(W, (hi.float() + lo.float()).cpu().numpy())
    Wd = dev(W, torch.bfloat16)
    got = rb.k_gemm(Wd, hi, impl=2, x_lo=lo).cpu().numpy()
    tol = 3e-5 * np.sqrt(K)
    np.testing.assert_allclose(got, want, rtol=0, atol=tol)
    assert np.array_equal(rb.k_gemm(Wd, hi, impl=2, x_lo=lo).cpu().numpy(), got)
    y0 = rng.normal(size=(M, N)).astype(np.float32)
    acc = rb.k_gemm(Wd, hi, y=dev(y0), accumulate=True, impl=2, x_lo=lo).cpu().numpy()
    np.testing.assert_allclose(acc, want + y0, rtol=0, atol=tol)


def _operand_pair(rng, M, K):
    x = dev(rng.normal(size=(M, K)).astype(np.float32))
    hi = x.to(torch.bfloat16)
    lo = (x - hi.float()).to(torch.bfloat16)
    return hi, lo, (hi.double() + lo.double()).cpu().numpy()


@pytest.mark.parametrize("M,N,K", [(1, 16, 64), (8, 576, 448), (3, 1536, 1536), (8, 512, 1408), (5, 3584, 3584), (2, 32, 8960)])
def test_rows_gemm_that_adds_into_the_residual(M, N, K):
    """The decode product of few rows that completes the residual stream: one chunk of K a warp, fewer chunks than warps, more than the
    ring's slots; the bound of the test above.  The operand and the sums of squares are exactly those of the y written."""
    rng = np.random.default_rng(M * 5 + N)
    W = ri.cpu_tensor(2, 9, N, K, True)
    hi, lo, x = _operand_pair(rng, M, K)
    y0 = rng.normal(size=(M, N)).astype(np.float32)
    gain = dev((1 + 0.1 * rng.normal(size=N)).astype(np.float32), torch.bfloat16)
    y = dev(y0)
    out_hi, out_lo, ssq = rb.k_gemm_rows(dev(W, torch.bfloat16), hi, lo, y, gain)
    np.testing.assert_allclose(y.cpu().numpy(), y0 + x @ W.astype(np.float64).T, rtol=0, atol=3e-5 * np.sqrt(K))
    v = y * gain.float()
    assert torch.equal(out_hi, v.to(torch.bfloat16)) and torch.equal(out_lo, (v - out_hi.float()).to(torch.bfloat16))
    want = (y.double() ** 2).view(M, N // 8, 8).sum(2)
    assert ((ssq.double() - want).abs() <= 8 * 2.0 ** -24 * want).all()          # eight roundings of positive terms


@pytest.mark.parametrize("M,N,K", [(8, 512, 1408), (1, 3584, 3584), (1, 512, 8960), (8, 16, 12288)])
def test_rows_gemm_rounds_no_more_than_a_k_split(M, N, K):
    """Against fp64 the product of few rows errs no more than the K split of the same operands.  An element's error varies, the norm over
    128 and more of them by 1 / sqrt(256) = 6 % at most; twice that is allowed."""
    rng = np.random.default_rng(K)
    W = dev(ri.cpu_tensor(2, 9, N, K, True), torch.bfloat16)
    hi, lo, x = _operand_pair(rng, M, K)
    exact = x @ W.double().cpu().numpy().T
    rows, split = torch.zeros(M, N, device="cuda"), torch.zeros(M, N, device="cuda")
    rb.k_gemm_rows(W, hi, lo, rows, torch.ones(N, dtype=torch.bfloat16, device="cuda"))
    rb.k_gemm(W, hi, y=split, accumulate=True, impl=2, x_lo=lo)
    errs = [np.linalg.norm(y.cpu().numpy() - exact) for y in (rows, split)]
    assert errs[0] <= 1.12 * errs[1], errs


@pytest.mark.parametrize("M,H,KV,hd,K,chunk,ext", [(1, 1, 1, 64, 64, 8, False), (8, 7, 1, 128, 576, 256, False), (3, 12, 2, 128, 1536, 8, True),
                                                   (5, 8, 8, 64, 512, 8, True)])
def test_rows_gemm_of_queries_keys_and_values(M, H, KV, hd, K, chunk, ext):
    """... and the one that ends in queries and cache pages: sums of squares per 8 and per 256 columns, first, last and middle slots of a
    page, one idle row, both caches.  The bound of the product grows by sqrt(2) where two values turn; keys and values carry fp16's rounding."""
    rng = np.random.default_rng(M + K)
    W = ri.cpu_tensor(2, 9, (H + 2 * KV) * hd, K, True)
    hi, lo, x = _operand_pair(rng, M, K)
    ssq = rng.uniform(0.5, 1.5, size=(M, -(-K // chunk))).astype(np.float32) * min(chunk, K)
    eps = 1e-6
    pos = np.array([15, 16, 40, 0, 33, 31, 7, 47][:M], np.int32)
    row = np.arange(M, dtype=np.int32)
    if M > 2:
        row[1] = -1
    table = rng.permutation(3 * M).reshape(M, 3).astype(np.int32)
    parts = 4 if ext else 2
    pool = torch.full((3 * M, parts, KV * 16 * hd), 7.0, dtype=torch.float16, device="cuda")
    ang = np.arange(48)[:, None] * 1e4 ** (-2.0 * np.arange(hd // 2) / hd)
    rope = np.stack([np.cos(ang), np.sin(ang)], -1).astype(np.float32)
    q = rb.k_gemm_rows_qkv(dev(W, torch.bfloat16), hi, lo, dev(ssq), eps, dev(row), dev(pos), dev(rope), pool, dev(table), H, KV, hd, ext)
    qkv = x @ W.astype(np.float64).T / np.sqrt(ssq.astype(np.float64).sum(1, keepdims=True) / K + eps)
    qkv = qkv.reshape(M, H + 2 * KV, hd)
    c, s = (rope[pos].astype(np.float64)[:, None, :, i] for i in (0, 1))
    a, b = qkv[:, :H + KV, :hd // 2].copy(), qkv[:, :H + KV, hd // 2:].copy()
    qkv[:, :H + KV, :hd // 2], qkv[:, :H + KV, hd // 2:] = a * c - b * s, b * c + a * s
    tol = 3e-5 * np.sqrt(2 * K)
    got = pool.cpu().numpy()
    touched = np.zeros(got.shape, bool)
    for m in range(M):
        if row[m] < 0:
            assert not q[m].any()
            continue
        np.testing.assert_allclose(q[m].cpu().numpy(), qkv[m, :H], rtol=0, atol=tol)
        pg, slot = table[m, pos[m] // 16], pos[m] % 16
        keys = [got[pg, i].reshape(KV, 16, hd)[:, slot].astype(np.float64) for i in range(0, parts, 2)]
        vals = [got[pg, i].reshape(KV, hd, 16)[:, :, slot].astype(np.float64) for i in range(1, parts, 2)]
        for i in range(parts):
            t = touched[pg, i].reshape((KV, hd, 16) if i & 1 else (KV, 16, hd))
            if i & 1:
                t[:, :, slot] = True
            else:
                t[:, slot] = True
        for have, want in ((sum(keys), qkv[m, H:H + KV]), (sum(vals), qkv[m, H + KV:])):
            np.testing.assert_allclose(have, want, rtol=2.0 ** (-21 if ext else -11), atol=tol + 2.0 ** -24)
    assert (got[~touched] == 7.0).all()


@pytest.mark.parametrize("M,N,K", [(2100, 2304, 3072), (2049, 2305, 3080), (512, 18944, 3136), (300, 18817, 3072), (4100, 1300, 1032)])
@pytest.mark.parametrize("kind", ["fp16", "bf16", "pairs"])
def test_dense_gemm_on_pairs_of_ctas(M, N, K, kind):
    """The paired kernel: one tile per pair and several, row and weight tiles that end ragged (also inside the leading CTA's
    half), a K tail, accumulation into y.  Against an fp32 product of the stored operands: fp32 sums of K products of
    N(0, 1) activations and N(0, 0.02) weights, bounded as in the tests above."""
    g = torch.Generator(device="cuda").manual_seed(M + N)
    W = torch.randn(N, K, generator=g, device="cuda") * 0.02
    x = torch.randn(M, K, generator=g, device="cuda")
    dt = torch.float16 if kind == "fp16" else torch.bfloat16
    Wd, hi = W.to(dt), x.to(dt)
    lo = (x - hi.float()).to(dt) if kind == "pairs" else None
    want = (hi.double() + (lo.double() if lo is not None else 0)) @ Wd.double().t()
    y = rb.k_gemm(Wd, hi, impl=4 if kind == "fp16" else 2, x_lo=lo)
    tol = 3e-5 * K ** 0.5
    assert (y.double() - want).abs().max().item() <= tol
    y2 = rb.k_gemm(Wd, hi, y=y.clone(), accumulate=True, impl=4 if kind == "fp16" else 2, x_lo=lo)
    assert (y2.double() - 2 * want).abs().max().item() <= 2 * tol


@pytest.mark.parametrize("M,F,K", [(1100, 1920, 3080), (300, 5056, 3072)])
def test_gate_up_gemm_on_pairs_of_ctas(M, F, K):
    """Plain gate/up tiles of the paired kernel, the last pair with one CTA's features missing: silu(g) * u rounded to bf16
    (2^-9 relative) after fp32 sums."""
    g = torch.Generator(device="cuda").manual_seed(M + F)
    W = (torch.randn(2 * F, K, generator=g, device="cuda") * 0.02).bfloat16()
    x = torch.randn(M, K, generator=g, device="cuda").bfloat16()
    act = torch.zeros(M, F, dtype=torch.bfloat16, device="cuda")
    nbytes = rb.lib().rsd_k_gemm_scratch_bytes(M, 2 * F, K)
    scratch = torch.zeros(nbytes, dtype=torch.uint8, device="cuda")
    assert rb.lib().rsd_k_gemm_gu(W.data_ptr(), x.data_ptr(), None, act.data_ptr(), None, M, F, K, scratch.data_ptr(), nbytes,
                                  torch.cuda.current_stream().cuda_stream) == 0
    gu = x.double() @ W.double().t()
    want = torch.nn.functional.silu(gu[:, :F]) * gu[:, F:]
    err = (act.double() - want).abs()
    assert (err <= 2 ** -8 * want.abs() + 3e-5 * K ** 0.5).all()
    assert int(scratch[4096:4100].view(torch.int32).item()) == 0


@pytest.mark.parametrize("M,N,K,adds", [(1100, 4608, 1024, False), (1290, 4500, 1032, False), (3000, 3584, 3080, True),
                                        (3200, 1536, 136, True), (4080, 1536, 136, True), (8100, 1530, 136, True)])
@pytest.mark.parametrize("dtype,impl", [(torch.float16, 4), (torch.bfloat16, 2)])
def test_dense_tiles_of_fewer_rows(M, N, K, adds, dtype, impl):
    """Products whose last wave of 256-row tiles would be nearly empty take tiles of 160, 192 and 224 rows, in pairs of CTAs (first three) and
    lone, of fp16 and of plain bf16 operands; ragged last tiles of rows and features.  fp32 sums of K products of order 0.05, as above."""
    g = torch.Generator(device="cuda").manual_seed(M + N)
    W = (torch.randn(N, K, generator=g, device="cuda") * 0.05).to(dtype)
    x = torch.randn(M, K, generator=g, device="cuda").to(dtype)
    y0 = torch.randn(M, N, generator=g, device="cuda")
    y = rb.k_gemm(W, x, y=y0.clone(), accumulate=True, impl=impl) if adds else rb.k_gemm(W, x, impl=impl)
    want = x.double() @ W.double().t() + (y0 if adds else 0)
    assert (y.double() - want).abs().max().item() <= 2e-5 * K ** 0.5 + 2e-6


@pytest.mark.parametrize("M,F,K", [(300, 2048, 136), (1300, 18944, 1024)])
def test_gate_up_tiles_of_fewer_rows(M, F, K):
    """The same for gate/up products: 160-row tiles of lone CTAs, 224-row tiles of pairs; the bound of the paired test above."""
    test_gate_up_gemm_on_pairs_of_ctas(M, F, K)


@pytest.mark.parametrize("one_pass", [0, 1])
def test_chunk_attention_wait_runs_out_cleanly(one_pass):
    """Failure path of the two tcgen05 chunk-attention kernels: no copy is issued, the bounded wait runs out, the flag is
    raised, nothing is written and the kernel returns (its tensor memory freed: the same kernel runs many times afterwards)."""
    rng = np.random.default_rng(41)
    T, H, KV = 16, 8, 1
    q = dev(rng.normal(size=(T, H, 128)).astype(np.float32))
    pool = torch.zeros(2 * 16 * 128, dtype=torch.float16, device="cuda")
    table = torch.zeros(1, dtype=torch.int32, device="cuda")
    row, pos = torch.zeros(T, dtype=torch.int32, device="cuda"), torch.arange(T, dtype=torch.int32, device="cuda")
    out = torch.full((T, H, 128), 7.0, device="cuda")
    flag = torch.zeros(1, dtype=torch.int32, device="cuda")
    stream = torch.cuda.current_stream().cuda_stream
    for _ in range(3):
        rc = rb.lib().rsd_debug_attn_wait_probe(one_pass, q.data_ptr(), pool.data_ptr(), table.data_ptr(), row.data_ptr(), pos.data_ptr(),
                                                out.data_ptr(), flag.data_ptr(), stream)
        assert rc == -5 and int(flag.item()) == -5
        assert b"bounded wait" in rb.lib().rsd_last_error(None)
        assert torch.all(out == 7.0)
    ctx = [700, 900] if one_pass else [100]           # 1600 entries x 24 heads (one pass) or 100 entries (two passes)
    H, KV = (24, 24) if one_pass else (8, 1)
    pool, table, Ks, Vs = paged_kv(rng, len(ctx), KV, 128, ctx, torch.float16, 64)
    rows = np.repeat(np.arange(len(ctx)), ctx).astype(np.int32)
    poss = np.concatenate([np.arange(c) for c in ctx]).astype(np.int32)
    qd = rng.normal(size=(len(rows), H, 128)).astype(np.float32)
    for _ in range(4):
        got = rb.k_attn_chunk(dev(qd), pool, table, dev(rows), dev(poss), KV).cpu().numpy()
    for t in (0, 50, len(rows) - 1):
        b, p = rows[t], poss[t]
        s = Ks[b][:p + 1, 0].astype(np.float64) @ qd[t, 0].astype(np.float64) / np.sqrt(128)
        w = np.exp(s - s.max()); w /= w.sum()
        np.testing.assert_allclose(got[t, 0], w @ Vs[b][:p + 1, 0].astype(np.float64), rtol=0, atol=2e-3)


# Rows of every instruction width and their edges; ids that leave no whole tile, one and some, a remainder of less than a piece, no multiple of
# four in the race; columns that do not fill a K step.
HEAD_SAMPLE = [(1, 515, 64, 515), (8, 4096, 72, 4001), (9, 1030, 768, 1030), (16, 38000, 520, 37999), (17, 75777, 64, 75777), (33, 40000, 1536, 39998),
               (64, 151936, 512, 151665), (65, 20000, 1536, 19999), (128, 38001, 264, 38001)]


@pytest.mark.parametrize("temperature", [0.0, 0.7])
@pytest.mark.parametrize("M,N,K,v_limit", HEAD_SAMPLE)
def test_head_that_samples(M, N, K, v_limit, temperature):
    """Against the head and the sampling one after the other: the sums are the same bits, so are the tokens.  Flat logits, logits with a peak, and two
    ids whose logits overflow (the lower one wins)."""
    gen = torch.Generator(device="cuda").manual_seed(M * N)
    W = torch.randn(N, K, generator=gen, device="cuda").mul_(0.05).to(torch.bfloat16)
    row = torch.randperm(M, generator=gen, device="cuda").to(torch.int32)
    if M > 1:
        row[M // 2] = -1
    pos = torch.randint(0, 500, (M,), generator=gen, device="cuda").to(torch.int32)
    ids = torch.randint(0, v_limit, (M,), generator=gen, device="cuda")
    flat = torch.randn(M, K, generator=gen, device="cuda")
    inputs = [(W, flat), (W, W[ids].float() * (20.0 / (0.0025 * K)))]
    huge = W.clone()
    huge[v_limit - 1] = 3e38
    huge[v_limit // 2] = 3e38
    inputs.append((huge, torch.full((M, K), 4.0, device="cuda")))
    for w, x in inputs:
        hi = x.to(torch.bfloat16)
        lo = (x - hi.float()).to(torch.bfloat16)
        got = rb.k_head_sample(w, hi, lo, v_limit, temperature, 77, 1, row, pos)
        logits = rb.k_gemm(w, hi, x_lo=lo, impl=3)
        want = rb.k_sample(logits, v_limit, temperature, 77, 1, row, pos)
        assert torch.equal(got, want), (got, want)
        if w is huge:
            assert (got[row >= 0] == v_limit // 2).all()


@pytest.mark.parametrize("score", [60.0, 1e3, 1e5, 1e7])
@pytest.mark.parametrize("M", [5, 16, 33, 128])
def test_head_that_samples_among_scores_that_tie(M, score):
    """Low temperatures: hundreds of ids share the largest logit and their scores differ by less than an ulp often, so the lowest of those that tie
    must win, whichever CTA comes first.  Against the sampling of the same logits, many positions, each several times."""
    gen = torch.Generator(device="cuda").manual_seed(M)
    N, K, v_limit = 50000, 64, 49990
    W = torch.zeros(N, K, device="cuda")
    same = torch.randperm(v_limit, generator=gen, device="cuda")[:3000]
    W[same, 0] = 4.0
    W[:, 1] = torch.randn(N, generator=gen, device="cuda")
    W = W.to(torch.bfloat16)
    W[same, 1] = 0
    hi = torch.zeros(M, K, dtype=torch.bfloat16, device="cuda")
    hi[:, 0] = 8.0
    hi[:, 1] = 0.5
    lo = torch.zeros_like(hi)
    row = torch.arange(M, dtype=torch.int32, device="cuda")
    logits = rb.k_gemm(W, hi, x_lo=lo, impl=3)
    for i in range(12):
        pos = torch.randint(0, 100000, (M,), generator=gen, device="cuda").to(torch.int32)
        want = rb.k_sample(logits, v_limit, 32.0 / score, 9, 2, row, pos)
        for _ in range(3):
            got = rb.k_head_sample(W, hi, lo, v_limit, 32.0 / score, 9, 2, row, pos)
            assert torch.equal(got, want), (i, (got != want).nonzero().flatten().tolist())


def test_head_that_samples_scales_its_rows():
    """The denominators of a norm ahead of the head, from sums of squares in one chunk and in many."""
    gen = torch.Generator(device="cuda").manual_seed(3)
    M, N, K = 24, 5000, 512
    W = torch.randn(N, K, generator=gen, device="cuda").mul_(0.05).to(torch.bfloat16)
    x = torch.randn(M, K, generator=gen, device="cuda") * torch.logspace(-1, 1, M, device="cuda")[:, None]
    hi = x.to(torch.bfloat16)
    lo = (x - hi.float()).to(torch.bfloat16)
    idx = torch.arange(M, device="cuda", dtype=torch.int32)
    logits = rb.k_gemm(W, hi, x_lo=lo, impl=3)
    for chunks in (2, 64):
        ssq = x.pow(2).view(M, chunks, -1).sum(-1)
        scaled = logits * torch.rsqrt(ssq.sum(-1, keepdim=True) / K + 1e-6)
        want = rb.k_sample(scaled, N, 0.7, 5, 0, idx, idx)
        got = rb.k_head_sample(W, hi, lo, N, 0.7, 5, 0, idx, idx, ssq=ssq.contiguous(), eps=1e-6)
        # the denominators' sums may differ in their last bits: a token may only where two scores are that close
        assert (got == want).float().mean() > 0.9


@pytest.mark.parametrize("chunks", [1, 3, 50, 129])
@pytest.mark.parametrize("M", [5, 16, 33, 128])
def test_head_that_samples_scales_its_rows_by_exact_denominators(M, chunks):
    """Sums of squares that are exact in any order and add up to a power of four a column: the denominators are powers of two, and so the scores, and the
    ids with them, are those of the scaled logits.  Chunks that the lanes of a row, 2 to 32 of them, do not share evenly."""
    gen = torch.Generator(device="cuda").manual_seed(M + chunks)
    N, K = 5000, 512
    W = torch.randn(N, K, generator=gen, device="cuda").mul_(0.05).to(torch.bfloat16)
    x = torch.randn(M, K, generator=gen, device="cuda")
    hi = x.to(torch.bfloat16)
    lo = (x - hi.float()).to(torch.bfloat16)
    idx = torch.arange(M, device="cuda", dtype=torch.int32)
    logits = rb.k_gemm(W, hi, x_lo=lo, impl=3)
    power = torch.randint(-2, 3, (M,), generator=gen, device="cuda").float()
    shares = torch.rand(M, chunks, generator=gen, device="cuda").mul_(900 / chunks).floor() + 1          # of 1024
    shares[:, chunks // 2] += 1024 - shares.sum(1)
    ssq = shares * (K / 1024) * torch.pow(4.0, power)[:, None]
    want = rb.k_sample(logits * torch.pow(2.0, -power)[:, None], N, 0.7, 5, 0, idx, idx)
    got = rb.k_head_sample(W, hi, lo, N, 0.7, 5, 0, idx, idx, ssq=ssq.contiguous(), eps=0.0)
    assert torch.equal(got, want)


def test_bounded_wait_runs_out_and_the_kernel_leaves_cleanly():
    """RSD_ERR_TIMEOUT without a fault: one CTA of the tensor-core GEMM whose copies are never issued.  Its wait
    (a few thousand polls in this mode) expires, the error flag is raised and reported, tensor memory is freed: the
    very next GEMMs on the same scratch are correct, many times over (a leaked allocation would stall them)."""
    rng = np.random.default_rng(5)
    W = dev(rng.normal(size=(128, 64)).astype(np.float32), torch.bfloat16)
    x = dev(rng.normal(size=(16, 64)).astype(np.float32), torch.bfloat16)
    y = torch.full((16, 128), 7.0, dtype=torch.float32, device="cuda")
    nbytes = rb.lib().rsd_k_gemm_scratch_bytes(16, 128, 64)
    scratch = torch.zeros(nbytes, dtype=torch.uint8, device="cuda")
    stream = torch.cuda.current_stream().cuda_stream
    for _ in range(3):
        rc = rb.lib().rsd_debug_gemm_wait_probe(W.data_ptr(), x.data_ptr(), y.data_ptr(), scratch.data_ptr(), nbytes, stream)
        assert rc == -5
        assert b"bounded wait" in rb.lib().rsd_last_error(None)
        assert int(scratch[4096:4100].view(torch.int32).item()) == 0           # cleared for the next use
        assert torch.all(y == 7.0)                                             # nothing was computed or written
    want = oracle.matmul(W.float().cpu().numpy(), x.float().cpu().numpy())
    for _ in range(40):                                  # 40 x 32 columns: more than the 512 a leak of 3 x 32 would leave
        got = torch.zeros(16, 128, dtype=torch.float32, device="cuda")
        assert rb.lib().rsd_k_gemm(W.data_ptr(), x.data_ptr(), None, got.data_ptr(), 16, 128, 64, 1, 0, 2, scratch.data_ptr(),
                                   nbytes, stream) == 0
        np.testing.assert_allclose(got.cpu().numpy(), want, rtol=0, atol=3e-4)
