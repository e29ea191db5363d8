"""The projection GEMM building block (tcgen05 / TMEM / TMA for bf16, SIMT
for fp32) against numpy fp64 matmul of the same bf16 operands, through the C
ABI (ravel_gemm).  Shapes cover single and multiple tiles, ragged token /
feature / K tails, split-K (partials exchanged through shared memory, or
through L2 for unaligned outputs), persistent launches on one SM
or on SM pairs (one 256-row MMA per K step across two CTAs) and every
epilogue."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def handles():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2609_34170_gb300 import build, ravel_create, ravel_destroy
    build.build()
    hs = {}
    for dt in ("bf16", "fp32"):
        cfg = synth.ExpertConfig(layers=1, width=64, n_q_heads=1, n_kv_heads=1, head_dim=64, mlp_dim=64, slots=2,
                                 action_dim=2, prefix=1, fop_tokens=0, batch=1, dtype=dt)
        hs[dt] = ravel_create(cfg, synth.make_weights(cfg))
    yield hs
    for h in hs.values():
        ravel_destroy(h)


def _rand(shape, seed, scale=1.0):
    return synth.round_bf16(np.random.default_rng(seed).standard_normal(shape).astype(np.float32) * scale)


SHAPES = [(1, 128, 64), (7, 100, 200), (50, 2560, 1024), (66, 1024, 2048), (50, 1024, 4096), (130, 384, 192),
          (300, 256, 512), (3200, 1024, 1024), (51, 3000, 1024), (4224, 2560, 1024), (3200, 1024, 2048),
          (3200, 1024, 4096), (2900, 2048, 704)]


@pytest.mark.parametrize("M,N,K", SHAPES)
@pytest.mark.parametrize("epi", [0, 1, 2])
def test_gemm_bf16(handles, M, N, K, epi):
    from paper_2609_34170_gb300 import ravel_gemm
    X, W = _rand((M, K), 1), _rand((N, K), 2, 0.05)
    bias = np.random.default_rng(3).standard_normal(N).astype(np.float32)
    ref = X.astype(np.float64) @ W.astype(np.float64).T + bias
    dev = lambda a, dt=torch.bfloat16: torch.from_numpy(a).to("cuda", dt)  # noqa: E731
    init = np.random.default_rng(4).standard_normal((M, N)).astype(np.float32)
    out = dev(init, torch.float32)
    ravel_gemm(handles["bf16"], dev(X), dev(W), epi, out, dev(bias, torch.float32))
    got = out.cpu().numpy().astype(np.float64)
    if epi == 1:
        ref = ref / (1 + np.exp(-ref))
    if epi == 2:
        ref = ref + init
    scale = np.sqrt(K) * 0.05 + 1
    np.testing.assert_allclose(got, ref, rtol=1e-4, atol=1e-4 * scale)


# Token counts between one robot's and many robots': every kind of plan (token
# tiles of 32 to 256, 1 to 8 splits with slices of 8 to 32 tokens, SM pairs with
# narrow tiles, several TMEM accumulators per item) with a ragged last tile.
# Tolerance: fp32 sums of K products of N(0, 1) and N(0, 0.05^2), as above.
@pytest.mark.parametrize("M", [33, 100, 137, 240, 431, 601, 1300, 1999])
@pytest.mark.parametrize("N,K", [(1024, 2048), (1024, 4096), (1536, 1024), (2500, 1032)])
def test_gemm_bf16_plans(handles, M, N, K):
    from paper_2609_34170_gb300 import ravel_gemm
    g = torch.Generator("cuda").manual_seed(M * N + K)
    X = torch.randn((M, K), generator=g, device="cuda").bfloat16()
    W = (torch.randn((N, K), generator=g, device="cuda") * 0.05).bfloat16()
    out = torch.randn((M, N), generator=g, device="cuda")
    ref = (X.double() @ W.double().T + out.double()).cpu().numpy()
    ravel_gemm(handles["bf16"], X, W, 2, out)
    scale = np.sqrt(K) * 0.05 + 1
    np.testing.assert_allclose(out.cpu().numpy(), ref, rtol=1e-4, atol=1e-4 * scale)
    half = torch.empty((M, N), device="cuda", dtype=torch.bfloat16)
    ravel_gemm(handles["bf16"], X, W, 0, half)
    np.testing.assert_allclose(half.float().cpu().numpy(), (X.double() @ W.double().T).cpu().numpy(), rtol=1e-2,
                               atol=1e-2 * scale)


# fp32 results against 64 bits, on each kind of plan: one K range per CTA, split
# and on SM pairs, with as many accumulators as k-tiles, fewer, and 9 (no power
# of two).  Bound: each of an accumulator's K / 16 truncating steps loses half an
# ulp (2^-24) of the sum, and the fp32 additions around them a few (what one
# accumulator gives at K = 4096, 4e-6, is above it wherever there are several).
@pytest.mark.parametrize("M,N,K", [(16, 128, 128), (50, 1024, 1024), (50, 1024, 4096), (240, 512, 560), (800, 1024, 4096),
                                   (1200, 1024, 4096), (1600, 1024, 4096), (3200, 1024, 1024), (431, 1025, 2048)])
@pytest.mark.parametrize("alloc", [True, False])
def test_gemm_fp32_results_are_short_sums(handles, M, N, K, alloc):
    from paper_2609_34170_gb300 import ravel_gemm, ravel_gemm_noalloc
    from tests.test_gemm_plans import SMS, load_plan
    g = torch.Generator("cuda").manual_seed(M + N + K)
    X = torch.randn((M, K), generator=g, device="cuda").bfloat16()
    W = (torch.randn((N, K), generator=g, device="cuda") * 0.02).bfloat16()
    out = torch.empty((M, N), device="cuda")
    if alloc:
        ravel_gemm(handles["bf16"], X, W, 0, out)
    else:
        ravel_gemm_noalloc(X, W, 0, out)
    p = load_plan()(M, N, K, 0, 0, 0, int(N % 4 == 0), (24 if alloc else 8) << 20)
    length = 64 * -(-((K + 63) // 64) // (p["splits"] * p["accs"]))
    ref = X.double() @ W.double().T
    err = float((out.double() - ref).norm() / ref.norm())
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    bound = ((length if sms == SMS else K) / 16 + 4) * 2.0 ** -24
    assert err < bound, (err, bound, p)


@pytest.mark.parametrize("M,N,K", [(50, 256, 1024), (50, 8192, 1024), (66, 4096, 1024), (66, 8192, 1024),
                                   (300, 1024, 256), (3200, 2048, 1024), (3200, 8192, 1024)])
@pytest.mark.parametrize("with_bias", [False, True])
def test_gemm_geglu_bf16(handles, M, N, K, with_bias):
    from paper_2609_34170_gb300 import ravel_gemm
    X, W = _rand((M, K), 5), _rand((N, K), 6, 0.05)
    bias = np.random.default_rng(9).standard_normal(N).astype(np.float32) if with_bias else np.zeros(N, np.float32)
    ref_all = X.astype(np.float64) @ W.astype(np.float64).T + bias   # bias of each gate / up row, before GELU
    blocks = ref_all.reshape(M, N // 128, 2, 64)
    g, u = blocks[:, :, 0].reshape(M, N // 2), blocks[:, :, 1].reshape(M, N // 2)
    ref = 0.5 * g * (1 + np.tanh(np.sqrt(2 / np.pi) * (g + 0.044715 * g ** 3))) * u
    out = torch.zeros((M, N // 2), device="cuda", dtype=torch.bfloat16)
    ravel_gemm(handles["bf16"], torch.from_numpy(X).to("cuda", torch.bfloat16),
               torch.from_numpy(W).to("cuda", torch.bfloat16), 3, out,
               torch.from_numpy(bias).cuda() if with_bias else None)
    got = out.float().cpu().numpy()
    np.testing.assert_allclose(got, ref, rtol=1e-2, atol=1e-2 * (np.abs(ref).max() + 1e-3))


# GeGLU of given gates (one product each, exact in fp32) on each kind of epilogue:
# one item per CTA, split slices, SM pairs and an unaligned output.  Bound: bf16's 8
# significant bits (2^-8 of the result) and tanh.approx's 2^-11 of tanh, times g / 2
# (the larger one for gates below -1.5, where 1 + tanh cancels).
@pytest.mark.parametrize("M,K,ld", [(4, 64, 1024), (50, 1024, 1024), (3200, 64, 1024), (50, 1024, 1028)])
def test_gemm_geglu_of_negative_gates(handles, M, K, ld):
    from paper_2609_34170_gb300 import _binding as B
    N = 2048
    gates = torch.linspace(-5, 5, N // 2, device="cuda").bfloat16()
    X = torch.zeros((M, K), device="cuda", dtype=torch.bfloat16)
    X[:, 0] = 1
    W = torch.zeros((N // 128, 2, 64, K), device="cuda", dtype=torch.bfloat16)
    W[:, 0, :, 0], W[:, 1, :, 0] = gates.view(-1, 64), 1
    out = torch.zeros((M, ld), device="cuda", dtype=torch.bfloat16)
    s = B.load().ravel_gemm(handles["bf16"], X.data_ptr(), M, K, K, W.data_ptr(), N, K, 3, out.data_ptr(), ld, 1, None,
                            torch.cuda.current_stream().cuda_stream)
    assert s == 0
    ref = torch.nn.functional.gelu(gates.double(), approximate="tanh")
    bound = ref.abs() * 2.0 ** -8 + gates.double().abs() * 2.0 ** -12 + 1e-6
    assert bool(((out[:, :N // 2].double() - ref).abs() <= bound).all())


def test_gemm_bf16_output_and_determinism(handles):
    from paper_2609_34170_gb300 import ravel_gemm
    M, N, K = 50, 1024, 4096      # split-K across the grid
    X, W = _rand((M, K), 7), _rand((N, K), 8, 0.05)
    Xd, Wd = torch.from_numpy(X).to("cuda", torch.bfloat16), torch.from_numpy(W).to("cuda", torch.bfloat16)
    outs = []
    for _ in range(3):
        o = torch.zeros((M, N), device="cuda", dtype=torch.bfloat16)
        ravel_gemm(handles["bf16"], Xd, Wd, 0, o)
        outs.append(o)
    assert all(torch.equal(outs[0], o) for o in outs[1:])
    ref = X.astype(np.float64) @ W.astype(np.float64).T
    np.testing.assert_allclose(outs[0].float().cpu().numpy(), ref, rtol=1e-2, atol=1e-2)


def test_gemm_two_sm_is_deterministic(handles):
    # the persistent two-SM kernel: every launch gives the same bits
    from paper_2609_34170_gb300 import ravel_gemm
    M, N, K = 3200, 1024, 4096
    X, W = _rand((M, K), 11), _rand((N, K), 12, 0.05)
    Xd, Wd = torch.from_numpy(X).to("cuda", torch.bfloat16), torch.from_numpy(W).to("cuda", torch.bfloat16)
    outs = []
    for _ in range(3):
        o = torch.zeros((M, N), device="cuda", dtype=torch.float32)
        ravel_gemm(handles["bf16"], Xd, Wd, 0, o)
        outs.append(o)
    assert all(torch.equal(outs[0], o) for o in outs[1:])
    ref = X.astype(np.float64) @ W.astype(np.float64).T
    np.testing.assert_allclose(outs[0].cpu().numpy(), ref, rtol=1e-4, atol=1e-4 * (np.sqrt(K) * 0.05 + 1))


# the row kernel: one ragged 8-row chunk, exact chunks, its last M and the
# first of the tile kernel; odd N, K that ends inside a lane's stride, and a K
# that is not whole float4s (the tile kernel); K split over warps with a ragged
# last step and row chunk, and either side of where that ends; either side of the
# lines on the products and on the rows
@pytest.mark.parametrize("M,N,K", [(1, 1, 4), (8, 16, 128), (10, 1027, 1024), (256, 33, 516), (257, 33, 516), (7, 40, 250),
                                   (5, 41, 516), (17, 300, 1024), (1, 1024, 512), (1, 1025, 512), (8, 1024, 508),
                                   (24, 30000, 64), (25, 30000, 64), (64, 8191, 512), (64, 8192, 512)])
@pytest.mark.parametrize("epi", [0, 1, 2])
def test_gemm_fp32_rows(handles, M, N, K, epi):
    from paper_2609_34170_gb300 import ravel_gemm
    g = torch.Generator("cuda").manual_seed(M + N + K)
    X, W = (torch.randn(s, generator=g, device="cuda") for s in ((M, K), (N, K)))
    bias, out = torch.randn(N, generator=g, device="cuda"), torch.randn((M, N), generator=g, device="cuda")
    ref = X.double() @ W.double().T + bias.double()
    ref = torch.nn.functional.silu(ref) if epi == 1 else ref + out.double() if epi == 2 else ref
    ravel_gemm(handles["fp32"], X, W, epi, out, bias)
    # K products of N(0, 1) values: |sum| errors below K 2^-24 sqrt(K)
    np.testing.assert_allclose(out.cpu().numpy(), ref.cpu().numpy(), rtol=1e-5, atol=max(1e-6, K ** 1.5 * 6e-8))


@pytest.mark.parametrize("M,N,K", [(10, 100, 256), (66, 300, 200)])
def test_gemm_fp32_simt(handles, M, N, K):
    from paper_2609_34170_gb300 import ravel_gemm
    rng = np.random.default_rng(9)
    X, W = rng.standard_normal((M, K)).astype(np.float32), rng.standard_normal((N, K)).astype(np.float32)
    out = torch.zeros((M, N), device="cuda")
    ravel_gemm(handles["fp32"], torch.from_numpy(X).cuda(), torch.from_numpy(W).cuda(), 0, out)
    np.testing.assert_allclose(out.cpu().numpy(), X.astype(np.float64) @ W.astype(np.float64).T, rtol=1e-5,
                               atol=1e-4)
