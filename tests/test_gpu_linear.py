"""GPU parity of a3 (block-scaled NVFP4 linear, tcgen05): outputs against the
oracle's fp64 product of identical dequantized operands.

Two kinds of inputs: (1) seeded random codes and scales handed to both sides
(isolates the GEMM from the quantizer), (2) the workloads' bf16 activations
and weights quantized by each side (codes are bit-exact, checked in
test_gpu_quantize), so the dequantized operands are identical."""
import numpy as np
import pytest
import torch

from _util import TOL, assert_close, assert_nvfp4_within, errors, f32, lib, swiglu_tolerance, u8
from oracle import nvfp4_oracle as O
from paper_2606_15682_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def N():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    return lib()


def random_operand(rows, K, gen, scale_lo=0x30, scale_hi=0x48):
    """Seeded random NVFP4 operand: packed codes, row-major scales (all codes, moderate scales)."""
    codes = torch.randint(0, 256, (rows, K // 2), generator=gen, dtype=torch.int32).to(torch.uint8).numpy()
    scales = torch.randint(scale_lo, scale_hi, (rows, K // 16), generator=gen, dtype=torch.int32).to(torch.uint8).numpy()
    return codes, scales


def run_linear(N, a_codes, a_scales_rm, g_a, w_codes, w_scales_rm, g_w, M, Nn, K, ldo=None):
    dev = "cuda"
    ac = torch.from_numpy(a_codes).to(dev)
    wc = torch.from_numpy(w_codes).to(dev)
    asf = torch.from_numpy(O.scales_to_mma(a_scales_rm)).to(dev)
    wsf = torch.from_numpy(O.scales_to_mma(w_scales_rm)).to(dev)
    ga = torch.tensor([g_a], dtype=torch.float32, device=dev)
    gw = torch.tensor([g_w], dtype=torch.float32, device=dev)
    ldo = Nn if ldo is None else ldo
    out = torch.full((M, ldo), float("nan"), dtype=torch.bfloat16, device=dev)
    N.nvfp4_linear(ac, asf, ga, wc, wsf, gw, out, M, Nn, K, ldo=ldo)
    torch.cuda.synchronize()
    assert N.nvfp4_get_device_status() == 0
    return out


@pytest.mark.parametrize("M,Nn,K", [(128, 128, 256), (1, 16, 256), (16, 128, 512), (130, 144, 512),
                                    (257, 384, 1024), (300, 272, 2304), (128, 1024, 256),
                                    # N % 256 == 0 with too few 256 x 256 tiles for the pairs and a short
                                    # K: single CTAs
                                    (256, 256, 512), (300, 512, 1024), (640, 768, 768), (129, 1280, 2048),
                                    (16, 1536, 1536), (256, 5120, 3584),
                                    # ... and with K >= 4096: split-K clusters of 2, 3 or 4 pairs, even
                                    # and uneven K ranges, M tails, a spare CTA per pair; M <= 128: the
                                    # skinny kernel
                                    (256, 512, 4096), (16, 1536, 4608), (1, 256, 4096), (300, 768, 5120),
                                    (100, 512, 6400), (256, 7168, 4096), (256, 5120, 4352),
                                    # CTA-pair path (enough 256 x 256 tiles to occupy the pairs):
                                    # M tails with a spare CTA, odd super-tile counts, one-row tail
                                    (256, 10240, 512), (300, 10240, 1024), (640, 5120, 768), (129, 12800, 256),
                                    # more 256 x 256 tiles than pairs: a second round of tiles, with an M
                                    # tail (K = 1536)
                                    (512, 10240, 1024), (300, 15360, 1536), (640, 7680, 1280),
                                    # N % 256 != 0 (CTA pairs with a column tail), and a pair shape with K = 4096
                                    # and a one-row M tail
                                    (640, 10112, 2048), (512, 10576, 2048), (257, 15360, 4096)])
def test_random_codes(N, M, Nn, K):
    gen = torch.Generator().manual_seed(M * 1000 + Nn * 10 + K)
    a_c, a_s = random_operand(M, K, gen)
    w_c, w_s = random_operand(Nn, K, gen)
    g_a, g_w = np.float32(0.0173), np.float32(0.00091)
    out = run_linear(N, a_c, a_s, g_a, w_c, w_s, g_w, M, Nn, K)
    ref = O.linear(a_c, a_s, g_a, w_c, w_s, g_w)
    assert_close(f32(out), ref, what=f"{M}x{Nn}x{K}")


@pytest.mark.parametrize("M,Nn,K,ldo", [(200, 160, 512, 200),     # single CTAs
                                        (200, 512, 4096, 520),    # split-K clusters
                                        (640, 10240, 1024, 10248)])  # CTA pairs
def test_ldo_padding_untouched(N, M, Nn, K, ldo):
    gen = torch.Generator().manual_seed(5)
    a_c, a_s = random_operand(M, K, gen)
    w_c, w_s = random_operand(Nn, K, gen)
    out = run_linear(N, a_c, a_s, 1.0, w_c, w_s, 1.0, M, Nn, K, ldo=ldo)
    ref = O.linear(a_c, a_s, 1.0, w_c, w_s, 1.0)
    assert_close(f32(out[:, :Nn]), ref)
    assert torch.isnan(out[:, Nn:].float()).all(), "columns beyond N must not be written"


def test_single_block_structure(N):
    # Only one nonzero 16-block per row: each output is one scaled block dot product,
    # so a misplaced scale (row, k-block) shows up as a wrong value.
    M, Nn, K = 128, 128, 512
    rng = np.random.default_rng(9)
    a_c = np.zeros((M, K // 2), np.uint8); w_c = np.zeros((Nn, K // 2), np.uint8)
    kb_a = rng.integers(0, K // 16, M); kb_w = rng.integers(0, K // 16, Nn)
    for r in range(M):
        a_c[r, kb_a[r] * 8:(kb_a[r] + 1) * 8] = rng.integers(0, 256, 8)
    for r in range(Nn):
        w_c[r, kb_w[r] * 8:(kb_w[r] + 1) * 8] = rng.integers(0, 256, 8)
    a_s = rng.integers(0x28, 0x50, (M, K // 16)).astype(np.uint8)
    w_s = rng.integers(0x28, 0x50, (Nn, K // 16)).astype(np.uint8)
    out = run_linear(N, a_c, a_s, 1.0, w_c, w_s, 1.0, M, Nn, K)
    ref = O.linear(a_c, a_s, 1.0, w_c, w_s, 1.0)
    assert_close(f32(out), ref)


@pytest.mark.parametrize("M,Nn,K", [(256, 256, 1024),    # single CTAs
                                    (256, 5120, 4352)])  # split-K clusters: partials summed in split order
def test_deterministic(N, M, Nn, K):
    gen = torch.Generator().manual_seed(11)
    # Wide scale range: partial sums that round in fp32, so a change of
    # summation order would show.
    a_c, a_s = random_operand(M, K, gen, 0x20, 0x58)
    w_c, w_s = random_operand(Nn, K, gen, 0x20, 0x58)
    o1 = run_linear(N, a_c, a_s, 1.0, w_c, w_s, 1.0, M, Nn, K)
    o2 = run_linear(N, a_c, a_s, 1.0, w_c, w_s, 1.0, M, Nn, K)
    assert torch.equal(o1, o2)


def quantize_gpu(N, x):
    g = torch.empty(1, dtype=torch.float32, device="cuda")
    N.nvfp4_tensor_scale(x, g)
    codes = torch.empty(x.shape[0], x.shape[1] // 2, dtype=torch.uint8, device="cuda")
    scales = torch.empty(N.nvfp4_scales_bytes(x.shape[0], x.shape[1], 1), dtype=torch.uint8, device="cuda")
    N.nvfp4_quantize(x, g, codes, scales, 1)
    return codes, scales, g


WL = [w for w in synth.WORKLOADS if "linears" in synth.WORKLOADS[w]]


@pytest.mark.parametrize("workload", WL)
def test_workload_linears(N, workload):
    """Every linear of every workload at full size, in the launch configuration the bench times.
    Large outputs are compared on seeded samples of rows and columns."""
    w = synth.WORKLOADS[workload]
    report = []
    for name, (Nn, K) in w["linears"].items():
        a, W = synth.linear_inputs(workload, name, device="cuda")
        M = a.shape[0]
        ac, asf, ga = quantize_gpu(N, a)
        wc, wsf, gw = quantize_gpu(N, W)
        out = torch.empty(M, Nn, dtype=torch.bfloat16, device="cuda")
        N.nvfp4_linear(ac, asf, ga, wc, wsf, gw, out, M, Nn, K)
        torch.cuda.synchronize()
        assert N.nvfp4_get_device_status() == 0
        rng = np.random.default_rng(1)
        rows = np.arange(M) if M * K <= 2048 * 8960 else np.sort(np.r_[rng.choice(M, 96, replace=False), M - 1])
        cols = np.arange(Nn) if Nn * K <= 17920 * 1536 else np.sort(np.r_[rng.choice(Nn, 256, replace=False), Nn - 1])
        g_a, g_w = O.tensor_scale(f32(a)), O.tensor_scale(f32(W))
        assert np.float32(ga.item()) == g_a and np.float32(gw.item()) == g_w
        ra_c, ra_s = O.quantize(f32(a[torch.as_tensor(rows, device="cuda")]), g_a)
        rw_c, rw_s = O.quantize(f32(W[torch.as_tensor(cols, device="cuda")]), g_w)
        ref = O.linear(ra_c, ra_s, g_a, rw_c, rw_s, g_w)
        got = f32(out[torch.as_tensor(rows, device="cuda")][:, torch.as_tensor(cols, device="cuda")])
        report.append((name,) + assert_close(got, ref, what=f"{workload}/{name}"))
    print(workload, report)


def test_injected_missing_stage_times_out_and_next_call_is_exact(N):
    """Failure detection of the GEMM without a GPU fault: the test-only fault
    knob makes both CTAs of the first CTA pair leave their first ring stage
    unissued.  The MMA issuer's and scale copiers' bounded waits run out after
    ~2 s, the pair drains its MMAs, frees TMEM and exits, the call reports
    NVFP4_ERR_TIMEOUT, and the next call is exact again."""
    import time
    M, Nn, K = 640, 10240, 2048  # a CTA-pair shape with more tiles than resident pairs
    gen = torch.Generator().manual_seed(31)
    a_c, a_s = random_operand(M, K, gen)
    w_c, w_s = random_operand(Nn, K, gen)
    dev = "cuda"
    args = (torch.from_numpy(a_c).to(dev), torch.from_numpy(O.scales_to_mma(a_s)).to(dev),
            torch.ones(1, device=dev), torch.from_numpy(w_c).to(dev),
            torch.from_numpy(O.scales_to_mma(w_s)).to(dev), torch.ones(1, device=dev))
    out = torch.full((M, Nn), float("nan"), dtype=torch.bfloat16, device=dev)
    torch.cuda.synchronize()
    assert N.nvfp4_get_device_status() == 0
    N.nvfp4_debug_inject_fault(N.FAULT_GEMM_SKIP_STAGE)
    try:
        t0 = time.time()
        N.nvfp4_linear(*args, out, M, Nn, K)
        torch.cuda.synchronize()
        waited = time.time() - t0
    finally:
        N.nvfp4_debug_inject_fault(N.FAULT_NONE)
    assert N.nvfp4_get_device_status() == 6
    assert 1.0 < waited < 20.0, f"bounded wait expected (~2-4 s), took {waited:.1f} s"
    out.fill_(float("nan"))
    N.nvfp4_linear(*args, out, M, Nn, K)
    torch.cuda.synchronize()
    assert N.nvfp4_get_device_status() == 0
    assert_close(f32(out), O.linear(a_c, a_s, 1.0, w_c, w_s, 1.0), what="after the injected timeout")


def test_injected_missing_stage_in_split_k_cluster_times_out(N):
    """The same fault in the split-K cluster kernel (a decode-sized shape with
    three CTA pairs per tile): the first pair of the first cluster leaves its
    first stage unissued; the other pairs of that cluster finish and wait at
    the cluster barrier, the faulted pair's bounded waits run out, the call
    reports NVFP4_ERR_TIMEOUT and the next call is exact."""
    import time
    M, Nn, K = 256, 5120, 4352
    gen = torch.Generator().manual_seed(37)
    a_c, a_s = random_operand(M, K, gen)
    w_c, w_s = random_operand(Nn, K, gen)
    dev = "cuda"
    args = (torch.from_numpy(a_c).to(dev), torch.from_numpy(O.scales_to_mma(a_s)).to(dev),
            torch.ones(1, device=dev), torch.from_numpy(w_c).to(dev),
            torch.from_numpy(O.scales_to_mma(w_s)).to(dev), torch.ones(1, device=dev))
    out = torch.full((M, Nn), float("nan"), dtype=torch.bfloat16, device=dev)
    torch.cuda.synchronize()
    assert N.nvfp4_get_device_status() == 0
    N.nvfp4_debug_inject_fault(N.FAULT_GEMM_SKIP_STAGE)
    try:
        t0 = time.time()
        N.nvfp4_linear(*args, out, M, Nn, K)
        torch.cuda.synchronize()
        waited = time.time() - t0
    finally:
        N.nvfp4_debug_inject_fault(N.FAULT_NONE)
    assert N.nvfp4_get_device_status() == 6
    assert 1.0 < waited < 20.0, f"bounded wait expected (~2-4 s), took {waited:.1f} s"
    out.fill_(float("nan"))
    N.nvfp4_linear(*args, out, M, Nn, K)
    torch.cuda.synchronize()
    assert N.nvfp4_get_device_status() == 0
    assert_close(f32(out), O.linear(a_c, a_s, 1.0, w_c, w_s, 1.0), what="after the injected timeout")


@pytest.mark.parametrize("M,Nn,K,swiglu", [(32, 1536, 5120, False),   # skinny, clusters that split K
                                           (128, 7168, 5120, False),
                                           (8, 5120, 2048, True),     # skinny, SwiGLU epilogue
                                           (300, 512, 1024, False)])  # single CTAs
def test_injected_missing_stage_in_the_other_gemm_kernels(N, M, Nn, K, swiglu):
    """The fault reaches whichever kernel serves the call and is spent there:
    the call reports NVFP4_ERR_TIMEOUT, the next one gives the same bytes as the
    one before the fault."""
    import time
    gen = torch.Generator().manual_seed(41)
    dev = "cuda"
    a_c, a_s = (torch.from_numpy(x).to(dev) for x in random_operand(M, K, gen))
    w_c, w_s = (torch.from_numpy(x).to(dev) for x in random_operand(Nn, K, gen))
    a_s, w_s = (torch.from_numpy(O.scales_to_mma(u8(x))).to(dev) for x in (a_s, w_s))
    g = torch.full((1,), 0.01, device=dev)

    def run():
        if swiglu:
            out = torch.full((M, Nn // 4), 0xEE, dtype=torch.uint8, device=dev)
            sc = torch.full((N.nvfp4_scales_bytes(M, Nn // 2, 1),), 0xEE, dtype=torch.uint8, device=dev)
            N.nvfp4_linear_swiglu_quantize(a_c, a_s, g, w_c, w_s, g, M, Nn // 2, K, g, out, sc)
            outs = (out, sc)
        else:
            outs = (torch.full((M, Nn), float("nan"), dtype=torch.bfloat16, device=dev),)
            N.nvfp4_linear(a_c, a_s, g, w_c, w_s, g, outs[0], M, Nn, K)
        torch.cuda.synchronize()
        return outs
    before = run()
    assert N.nvfp4_get_device_status() == 0
    N.nvfp4_debug_inject_fault(N.FAULT_GEMM_SKIP_STAGE)
    try:
        t0 = time.time()
        run()
        waited = time.time() - t0
        assert N.nvfp4_get_device_status() == 6
        assert 1.0 < waited < 20.0, f"bounded wait expected (~2-4 s), took {waited:.1f} s"
        after = run()
        assert N.nvfp4_get_device_status() == 0
    finally:
        N.nvfp4_debug_inject_fault(N.FAULT_NONE)
    assert all(torch.equal(x, y) for x, y in zip(before, after))


# ------------------------------------ gate_up with SwiGLU + quantize fused ---

def test_interleave_gate_up_matches_oracle(N):
    gen = torch.Generator().manual_seed(12)
    I, K = 96, 200
    g = torch.randn(I, K, generator=gen).to(torch.bfloat16)
    u = torch.randn(I, K, generator=gen).to(torch.bfloat16)
    out = torch.empty(2 * I, K, dtype=torch.bfloat16, device="cuda")
    N.nvfp4_interleave_gate_up(g.cuda(), u.cuda(), out)
    torch.cuda.synchronize()
    ref = O.interleave_gate_up(g.view(torch.int16).numpy(), u.view(torch.int16).numpy())
    assert np.array_equal(out.cpu().view(torch.int16).numpy(), ref)


def swiglu_case(N, M, I, K, seed, rows=None):
    gen = torch.Generator().manual_seed(seed)
    a_c, a_s = random_operand(M, K, gen)
    wg_c, wg_s = random_operand(I, K, gen, 0x30, 0x40)
    wu_c, wu_s = random_operand(I, K, gen, 0x30, 0x40)
    g_a, g_w = np.float32(0.0173), np.float32(0.0021)
    rows = np.arange(M) if rows is None else rows
    G = O.linear_rows(a_c, a_s, g_a, wg_c, wg_s, g_w, rows)
    U = O.linear_rows(a_c, a_s, g_a, wu_c, wu_s, g_w, rows)
    h = O.silu(G) * U
    g_out = O.tensor_scale(h.astype(np.float32))            # a calibrated static scale
    w_c = O.interleave_gate_up(wg_c, wu_c)
    w_s = O.interleave_gate_up(wg_s, wu_s)
    dev = "cuda"
    out_c = torch.full((M, I // 2), 0xEE, dtype=torch.uint8, device=dev)
    out_s = torch.full((N.nvfp4_scales_bytes(M, I, 1),), 0xEE, dtype=torch.uint8, device=dev)
    N.nvfp4_linear_swiglu_quantize(torch.from_numpy(a_c).to(dev), torch.from_numpy(O.scales_to_mma(a_s)).to(dev),
                                   torch.tensor([g_a], device=dev), torch.from_numpy(w_c).to(dev),
                                   torch.from_numpy(O.scales_to_mma(w_s)).to(dev), torch.tensor([g_w], device=dev),
                                   M, I, K, torch.tensor([g_out], device=dev), out_c, out_s)
    torch.cuda.synchronize()
    assert N.nvfp4_get_device_status() == 0
    return h, g_out, rows, u8(out_c), u8(out_s), swiglu_tolerance(G, U, h)


@pytest.mark.parametrize("M,I,K", [(256, 128, 256), (129, 384, 512), (300, 256, 1024), (640, 512, 768),
                                  # last waves in half tiles (76 pairs): 78 and 40 + 76 tiles
                                  (300, 4992, 768), (256, 14848, 512)])
def test_linear_swiglu_quantize(N, M, I, K):
    """h = SiLU(gate) * up from the fp32 accumulators, quantized with a static
    scale.  The kernel's SiLU uses the hardware tanh approximation, so every
    block scale and code must be one the recipe gives for some h' within that
    approximation's error of the exact fp64 h; no other difference is allowed.
    Most equal the oracle's quantization of h; padding scales are zero."""
    h, g_out, rows, out_c, out_s, tol = swiglu_case(N, M, I, K, seed=M + I + K)
    rc, rs = O.quantize(h.astype(np.float32), g_out)
    gs = O.scales_from_mma(out_s, M, I)
    assert_nvfp4_within(out_c, gs, h, tol, g_out, what=f"swiglu {M}x{I}x{K}")
    assert (gs == rs).mean() > 0.99 and (out_c == rc).mean() > 0.99
    pad = np.setdiff1d(np.arange(O.mma_scale_bytes(M, I)), O._mma_offsets(M, I // 16).ravel())
    assert not out_s[pad].any(), "padding rows of the output scales must be zero"


def test_linear_swiglu_quantize_prefill_shape_then_down(N):
    """The 1.5B-prefill MLP shape (M=2048, I=8960, K=1536) checked on sampled rows,
    then fed to the down projection as its A operand."""
    M, I, K, Hd = 2048, 8960, 1536, 1536
    rows = np.sort(np.r_[np.random.default_rng(2).choice(M, 48, replace=False), M - 1])
    h, g_out, rows, out_c, out_s, tol = swiglu_case(N, M, I, K, seed=99, rows=rows)
    gs = O.scales_from_mma(out_s, M, I)[rows]
    assert_nvfp4_within(out_c[rows], gs, h, tol, g_out, what="swiglu 1.5B prefill")
    # down projection straight from the fused output
    gen = torch.Generator().manual_seed(7)
    wd_c, wd_s = random_operand(Hd, I, gen)
    g_wd = np.float32(0.003)
    out = torch.empty(M, Hd, dtype=torch.bfloat16, device="cuda")
    N.nvfp4_linear(torch.from_numpy(out_c).cuda(), torch.from_numpy(out_s).cuda(),
                   torch.tensor([g_out], device="cuda"), torch.from_numpy(wd_c).cuda(),
                   torch.from_numpy(O.scales_to_mma(wd_s)).cuda(), torch.tensor([g_wd], device="cuda"), out, M, Hd, I)
    torch.cuda.synchronize()
    assert N.nvfp4_get_device_status() == 0
    ref = O.linear_rows(out_c, O.scales_from_mma(out_s, M, I), g_out, wd_c, wd_s, g_wd, rows)
    assert_close(f32(out[torch.as_tensor(rows, device="cuda")]), ref, what="down(swiglu)")


@pytest.mark.parametrize("M,I,K", [(1, 128, 256), (3, 20480, 512), (8, 256, 1280), (31, 384, 1024),
                                   (32, 128, 4096), (5, 128, 4352), (33, 256, 768), (33, 9856, 512), (64, 6144, 512),
                                   (65, 9856, 256), (128, 10240, 512)])
@pytest.mark.parametrize("fmt", ["nvfp4", "mxfp4", "mxfp4_rot"])
def test_linear_swiglu_quantize_few_rows(N, M, I, K, fmt):
    """Up to 128 rows run in a kernel of their own for some shapes, with the same sums and the
    same epilogue arithmetic as the CTA pairs: its codes and scales equal, byte
    for byte, those that the pairs give these rows within a taller activation,
    and the scales of its padding rows those of zeros."""
    dev, tall = "cuda", 256
    gen = torch.Generator(device=dev)
    gen.manual_seed(M + I + K)

    def operand(rows):
        lo, hi = (0x30, 0x40) if fmt == "nvfp4" else (122, 128)
        return (torch.randint(0, 256, (rows, K // 2), dtype=torch.uint8, device=dev, generator=gen),
                torch.randint(lo, hi, (N.nvfp4_scales_bytes(rows, K, 1),), dtype=torch.uint8, device=dev, generator=gen))

    (a_c, a_s), (w_c, w_s) = operand(tall), operand(2 * I)
    if fmt != "nvfp4":
        # MXFP4 scales: a byte for each 16-element half of a 32-element block, both equal.
        a_s[1::2], w_s[1::2] = a_s[::2], w_s[::2]
    g, g_out = torch.full((1,), 0.05, device=dev), torch.full((1,), 1e-2, device=dev)

    def run(rows):
        out_c = torch.full((rows, I // 2), 0xEE, dtype=torch.uint8, device=dev)
        out_s = torch.full((N.nvfp4_scales_bytes(rows, I, 1),), 0xEE, dtype=torch.uint8, device=dev)
        if fmt == "nvfp4":
            N.nvfp4_linear_swiglu_quantize(a_c, a_s, g, w_c, w_s, g, rows, I, K, g_out, out_c, out_s)
        else:
            N.mxfp4_linear_swiglu_quantize(a_c, a_s, w_c, w_s, rows, I, K, out_c, out_s, rotate=fmt == "mxfp4_rot")
        torch.cuda.synchronize()
        assert N.nvfp4_get_device_status() == 0
        return u8(out_c), O.scales_from_mma(u8(out_s), max(rows, 128), I)

    (codes, scales), (want_c, want_s) = run(M), run(tall)
    assert (codes == want_c[:M]).all() and (scales[:M] == want_s[:M]).all()
    assert len(np.unique(codes)) > 8
    assert not scales[M:].any()


@pytest.mark.parametrize("M", [256, 20])  # CTA pairs, skinny kernel
def test_linear_swiglu_quantize_invalid_g_out_zeroes_and_reports(N, M):
    I, K = 128, 256
    gen = torch.Generator().manual_seed(3)
    a_c, a_s = random_operand(M, K, gen)
    w_c, w_s = random_operand(2 * I, K, gen)
    dev = "cuda"
    out_c = torch.full((M, I // 2), 0xEE, dtype=torch.uint8, device=dev)
    out_s = torch.full((N.nvfp4_scales_bytes(M, I, 1),), 0xEE, dtype=torch.uint8, device=dev)
    N.nvfp4_get_device_status()
    N.nvfp4_linear_swiglu_quantize(torch.from_numpy(a_c).to(dev), torch.from_numpy(O.scales_to_mma(a_s)).to(dev),
                                   torch.ones(1, device=dev), torch.from_numpy(w_c).to(dev),
                                   torch.from_numpy(O.scales_to_mma(w_s)).to(dev), torch.ones(1, device=dev),
                                   M, I, K, torch.tensor([-1.0], device=dev), out_c, out_s)
    torch.cuda.synchronize()
    assert N.nvfp4_get_device_status() == 1
    assert not u8(out_c).any() and not u8(out_s).any()


@pytest.mark.parametrize("M,Nn,K,ldo", [
    # the skinny kernel (one row tile): A box and slot edges, N tails, each split, uneven K ranges
    (1, 16, 1792, 16), (8, 112, 2048, 120), (9, 144, 2304, 144), (31, 272, 4864, 280), (32, 5136, 1792, 5136),
    (33, 1536, 2304, 1536), (63, 2064, 4096, 2064), (64, 7168, 2560, 7168), (65, 1296, 5120, 1304),
    (127, 10240, 2560, 10240), (128, 256, 10240, 256), (5, 14352, 2048, 14352), (17, 20000, 1536, 20000),
    (128, 20480, 2304, 20480), (32, 28048, 1792, 28048), (1, 128, 27648, 128)])
def test_skinny_shapes(N, M, Nn, K, ldo):
    gen = torch.Generator().manual_seed(M * 1000 + Nn * 10 + K)
    a_c, a_s = random_operand(M, K, gen)
    w_c, w_s = random_operand(Nn, K, gen)
    g_a, g_w = np.float32(0.0173), np.float32(0.00091)
    out = run_linear(N, a_c, a_s, g_a, w_c, w_s, g_w, M, Nn, K, ldo=ldo)
    ref = O.linear(a_c, a_s, g_a, w_c, w_s, g_w)
    assert_close(f32(out[:, :Nn]), ref, what=f"{M}x{Nn}x{K}")
    assert torch.isnan(out[:, Nn:].float()).all()
    again = run_linear(N, a_c, a_s, g_a, w_c, w_s, g_w, M, Nn, K, ldo=ldo)
    assert torch.equal(out[:, :Nn], again[:, :Nn])


def test_skinny_reads_a_weight_written_by_the_kernel_before_it(N):
    """The skinny kernel prefetches W into L2 before the preceding kernel has
    finished; a W that this kernel writes must be read as written."""
    M, Nn, K = 4, 7168, 2560
    gen = torch.Generator(device="cuda").manual_seed(3)
    x = torch.randn(M, K, generator=gen, device="cuda").to(torch.bfloat16)
    ws = [(torch.randn(Nn, K, generator=gen, device="cuda") * s).to(torch.bfloat16) for s in (0.02, 0.5)]
    new = lambda *s, dtype=torch.uint8: torch.zeros(*s, dtype=dtype, device="cuda")  # noqa: E731
    ac, asf, g = new(M, K // 2), new(N.nvfp4_scales_bytes(M, K, 1)), new(1, dtype=torch.float32)
    wc, wsf, gw = new(Nn, K // 2), new(N.nvfp4_scales_bytes(Nn, K, 1)), new(1, dtype=torch.float32)
    outs = [new(M, Nn, dtype=torch.bfloat16) for _ in range(4)]
    N.nvfp4_tensor_scale(x, g)
    N.nvfp4_quantize(x, g, ac, asf)
    gw.fill_(0.001)
    for i in range(4):
        if i >= 2:
            torch.cuda.synchronize()
        N.nvfp4_quantize(ws[i % 2], gw, wc, wsf)
        if i >= 2:
            torch.cuda.synchronize()
        N.nvfp4_linear(ac, asf, g, wc, wsf, gw, outs[i], M, Nn, K)
    torch.cuda.synchronize()
    assert N.nvfp4_get_device_status() == 0
    assert torch.equal(outs[0], outs[2]) and torch.equal(outs[1], outs[3]) and not torch.equal(outs[0], outs[1])


@pytest.mark.parametrize("M,Nn,K", [
    # last waves whose tiles are split into 256 x 128 halves (76 pairs): only halves, after one
    # full wave, with M tails and a spare CTA, two k-blocks and more than the ring's
    (256, 9728, 512), (300, 9984, 768), (256, 27648, 1024), (1000, 5120, 2048), (130, 19712, 1792)])
def test_last_wave_in_half_tiles(N, M, Nn, K):
    gen = torch.Generator().manual_seed(M * 1000 + Nn * 10 + K)
    a_c, a_s = random_operand(M, K, gen)
    w_c, w_s = random_operand(Nn, K, gen)
    g_a, g_w = np.float32(0.0173), np.float32(0.00091)
    out = run_linear(N, a_c, a_s, g_a, w_c, w_s, g_w, M, Nn, K, ldo=Nn + 8)
    ref = O.linear(a_c, a_s, g_a, w_c, w_s, g_w)
    assert_close(f32(out[:, :Nn]), ref, what=f"{M}x{Nn}x{K}")
    assert torch.isnan(out[:, Nn:].float()).all()


@pytest.mark.parametrize("M,Nn,K,ldo", [
    # CTA pairs with a column tail: inside the first and the second half of the last tile, one
    # 16-column chunk, with half tiles in the last wave, an M tail and a padded pitch
    (300, 10000, 1792, 10000), (130, 19472, 2304, 19480), (640, 7312, 2048, 7312), (1000, 2576, 4096, 2584),
    (2000, 1296, 2304, 1296), (600, 15376, 1536, 15376)])
def test_pair_column_tails(N, M, Nn, K, ldo):
    gen = torch.Generator().manual_seed(M * 1000 + Nn * 10 + K)
    a_c, a_s = random_operand(M, K, gen)
    w_c, w_s = random_operand(Nn, K, gen)
    g_a, g_w = np.float32(0.0173), np.float32(0.00091)
    out = run_linear(N, a_c, a_s, g_a, w_c, w_s, g_w, M, Nn, K, ldo=ldo)
    ref = O.linear(a_c, a_s, g_a, w_c, w_s, g_w)
    assert_close(f32(out[:, :Nn]), ref, what=f"{M}x{Nn}x{K}")
    assert torch.isnan(out[:, Nn:].float()).all()
