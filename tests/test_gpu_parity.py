"""GPU parity of the rolling step against the fp64 oracle, through the C ABI.

Tolerances (fixed for the step): fp32 mode released max-abs <= 1e-4 and
velocity relative L2 <= 1e-4; bf16 mode 5e-2 and 2e-2; the appended Gaussian
slot bit-exact in both modes.
"""
import numpy as np
import pytest

import synth
from oracle import expert, noise
from tests._harness import TOL, Case, check_step, gpu_session, oracle_step, rel_l2

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2609_34170_gb300 import build, load
    build.build()
    load()


def _ragged(dtype, **kw):
    base = dict(layers=2, width=192, n_q_heads=6, n_kv_heads=2, head_dim=40, mlp_dim=320, slots=7,
                action_dim=5, prefix=45, fop_tokens=3, batch=3, dtype=dtype)
    base.update(kw)
    return synth.ExpertConfig(**base)


def test_reset_noise_bit_exact_over_a_million_draws():
    cfg = synth.ExpertConfig(layers=1, width=64, n_q_heads=1, n_kv_heads=1, head_dim=64, mlp_dim=64, slots=50,
                             action_dim=31, prefix=1, fop_tokens=0, batch=700, dtype="fp32")
    seeds = np.array([(b * 0x9E3779B97F4A7C15 + 17) % 2 ** 64 for b in range(cfg.batch)], dtype=np.uint64)
    from paper_2609_34170_gb300 import RollingSession
    s = RollingSession(cfg, synth.make_weights(cfg), 0)
    s.reset(seeds)
    got = s.buffer.cpu().numpy()
    want, cnt = expert.reset(cfg, seeds)
    assert got.size >= 10 ** 6
    np.testing.assert_array_equal(got, want)
    np.testing.assert_array_equal(s.counters(), cnt)
    s.close()


def test_tiny_fp32_single_step_and_rollout():
    cfg = synth.PRESETS["tiny_fp32_b1"]
    case = Case(cfg)
    s = gpu_session(case)
    for i in range(21):   # one step plus a 20-step rollout, teacher-forced
        check_step(case, s, label=f"step {i}")
    s.close()


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
def test_ragged_shapes(dtype):
    cfg = _ragged(dtype)
    case = Case(cfg, prefix_len=37)           # prefix shorter than the slot capacity
    s = gpu_session(case, max_batch=4, max_prefix=cfg.prefix)
    for i in range(3):
        check_step(case, s, label=f"{dtype} step {i}")
    s.close()


# Key chunks split over a thread-block cluster (2, 4, 16 splits; one and two
# query tiles; two robots), with a partial last prefix chunk, and a prefix
# shorter than the slot capacity so that some splits get no key at all; and
# head dims that are not a multiple of 64.
SPLIT_KV = [
    (dict(layers=2, width=256, n_q_heads=4, n_kv_heads=1, head_dim=64, mlp_dim=512, slots=20, action_dim=7,
          prefix=300, fop_tokens=5, batch=1), None),
    (dict(layers=2, width=256, n_q_heads=4, n_kv_heads=2, head_dim=128, mlp_dim=512, slots=12, action_dim=5,
          prefix=700, fop_tokens=4, batch=1), None),
    (dict(layers=1, width=256, n_q_heads=2, n_kv_heads=1, head_dim=128, mlp_dim=256, slots=12, action_dim=5,
          prefix=2000, fop_tokens=3, batch=1), 1500),
    (dict(layers=1, width=256, n_q_heads=8, n_kv_heads=2, head_dim=64, mlp_dim=256, slots=40, action_dim=6,
          prefix=500, fop_tokens=8, batch=2), None),
    # head dims that end inside a 64-wide block: P V reads V as an MN-major
    # operand whose second block is partial (96 = 64 + 32 split, 80 = 64 + 16
    # over 64 robots, whose query tiles are not split)
    (dict(layers=1, width=192, n_q_heads=4, n_kv_heads=2, head_dim=96, mlp_dim=256, slots=10, action_dim=5,
          prefix=260, fop_tokens=3, batch=1), None),
    (dict(layers=1, width=160, n_q_heads=2, n_kv_heads=1, head_dim=80, mlp_dim=256, slots=9, action_dim=4,
          prefix=130, fop_tokens=2, batch=64), None),
]


@pytest.mark.parametrize("kw,prefix_len", SPLIT_KV)
def test_split_kv_attention(kw, prefix_len):
    cfg = synth.ExpertConfig(**kw, dtype="bf16")
    case = Case(cfg, prefix_len=prefix_len)
    s = gpu_session(case)
    for i in range(2):
        check_step(case, s, label=f"split-kv step {i}")
    s.close()


def test_slot_isolated_mask():
    cfg = _ragged("fp32", batch=2)
    case = Case(cfg)
    s = gpu_session(case, mask_mode=1)
    check_step(case, s, mask="slot_isolated")
    s.close()


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
def test_no_fop_tokens(dtype):
    cfg = _ragged(dtype, fop_tokens=0, batch=2)
    case = Case(cfg)
    s = gpu_session(case)
    check_step(case, s)
    s.close()


def test_context_swap_and_errors():
    from paper_2609_34170_gb300 import RavelError, RollingSession
    cfg = _ragged("fp32", batch=2)
    a = Case(cfg)
    b = Case(cfg, ctx_seed=555, prefix_len=20)
    s = RollingSession(cfg, a.W, 0, 2, cfg.prefix)
    s.reset(a.seeds)
    with pytest.raises(RavelError) as ei:
        s.step(a.t, a.fop, a.delta)
    assert ei.value.status == 5                   # no context yet
    with pytest.raises(RavelError) as ei:
        s.set_context(a.k, a.v, cfg.prefix + 1)
    assert ei.value.status == 2                   # prefix too long
    s.set_context(a.k, a.v, a.P)
    with pytest.raises(RavelError) as ei:
        s.set_context(b.k, b.v, b.P)
    assert ei.value.status == 6                   # previous swap still pending
    check_step(a, s, label="context A")
    side = torch.cuda.Stream()
    s.set_context(b.k, b.v, b.P, side_stream=side)   # swapped in from a side stream
    check_step(b, s, label="context B")
    check_step(b, s, label="context B reused")
    s.close()


def test_state_resume_is_bit_exact():
    cfg = _ragged("bf16", batch=2)
    case = Case(cfg)
    s = gpu_session(case)
    for _ in range(3):
        s.step(case.t, case.fop, case.delta)
    saved_buf, saved_cnt = s.buffer.clone(), s.counters()
    outs = [s.step(case.t, case.fop, case.delta).clone() for _ in range(4)]
    s.buffer.copy_(saved_buf)
    s.set_counters(saved_cnt)
    again = [s.step(case.t, case.fop, case.delta).clone() for _ in range(4)]
    for x, y in zip(outs, again):
        assert torch.equal(x, y)
    s.close()


@pytest.mark.parametrize("name,robots", [("pi05_bf16_b1", [0]), ("pi05_bf16_b64", [0, 37, 63]),
                                         ("wide_bf16_b8", [0, 5, 7])])
def test_full_size_configs_sampled(name, robots):
    cfg = synth.PRESETS[name]
    case = Case(cfg)
    s = gpu_session(case)
    check_step(case, s, robots=robots, label=name)
    s.close()


# Chunks of 128 keys in two halves: prefixes that end inside the first or the
# second half, at their edges and one key past them, own keys (slots + FOP) in
# one and two halves and chunks, unsplit (many robots) and split; capacities
# above the prefix.
@pytest.mark.parametrize("prefix,capacity", [(1, 1), (63, 200), (64, 64), (65, 129), (127, 128), (128, 384), (129, 700)])
@pytest.mark.parametrize("batch,slots,fop", [(1, 50, 16), (40, 20, 4), (2, 130, 3)])
def test_attention_chunk_edges(prefix, capacity, batch, slots, fop):
    cfg = synth.ExpertConfig(layers=1, width=128, n_q_heads=4, n_kv_heads=2, head_dim=64, mlp_dim=128, slots=slots,
                             action_dim=4, prefix=capacity, fop_tokens=fop, batch=batch, dtype="bf16")
    case = Case(cfg, prefix_len=prefix)
    s = gpu_session(case)
    check_step(case, s, robots=sorted({0, batch // 2, batch - 1}), label=f"prefix {prefix}")
    s.close()


# The fp32 attention: head dims at the edges of its column groups (8 columns, a
# whole and a part group of 64, 128 and 256), keys that fill a chunk of 32, end
# one past it and span several.
@pytest.mark.parametrize("hd", [8, 64, 72, 128, 136, 256])
@pytest.mark.parametrize("prefix,slots,fop", [(24, 5, 3), (25, 5, 3), (70, 17, 0)])
@pytest.mark.parametrize("mask", ["full", "slot_isolated"])
def test_fp32_attention_edges(hd, prefix, slots, fop, mask):
    cfg = synth.ExpertConfig(layers=1, width=64, n_q_heads=6, n_kv_heads=2, head_dim=hd, mlp_dim=64, slots=slots,
                             action_dim=3, prefix=prefix, fop_tokens=fop, batch=2, dtype="fp32")
    s = gpu_session(Case(cfg), mask_mode=int(mask != "full"))
    check_step(Case(cfg), s, mask=mask, label=f"head dim {hd}")
    s.close()


# fp32 GeGLU in the row kernel: part and whole row chunks, the last row count it
# takes and the first that goes through the separate launch, one and several
# gate/up groups, widths on either side of the split of K.
@pytest.mark.parametrize("batch,slots", [(1, 2), (3, 3), (8, 32), (1, 257)])
@pytest.mark.parametrize("width,mlp", [(64, 64), (512, 192), (520, 1024)])
def test_fp32_geglu_rows(batch, slots, width, mlp):
    cfg = synth.ExpertConfig(layers=2, width=width, n_q_heads=2, n_kv_heads=1, head_dim=16, mlp_dim=mlp, slots=slots,
                             action_dim=3, prefix=9, fop_tokens=2, batch=batch, dtype="fp32")
    s = gpu_session(Case(cfg))
    check_step(Case(cfg), s, robots=sorted({0, batch - 1}), label=f"rows {batch * slots}")
    s.close()


# The fused head and tail: action widths at the edges of a noise group and of its
# 32 outputs, one and several passes over the row, a slot per CTA: few and many.
@pytest.mark.parametrize("batch,slots", [(1, 2), (5, 9), (1, 152)])
@pytest.mark.parametrize("width,actions", [(64, 1), (1024, 20), (1032, 32), (2056, 5)])
def test_head_tail_edges(batch, slots, width, actions):
    cfg = synth.ExpertConfig(layers=1, width=width, n_q_heads=2, n_kv_heads=1, head_dim=64, mlp_dim=64, slots=slots,
                             action_dim=actions, prefix=9, fop_tokens=2, batch=batch, dtype="bf16")
    case = Case(cfg)
    s = gpu_session(case)
    for _ in range(2):   # (the second step starts from the first one's buffer and counters)
        check_step(case, s, label=f"{batch * slots} rows")
    s.close()


# The same for more rows than two per SM, where a CTA takes eight slots of a
# robot: whole and ragged groups of slots, fewer than eight, one and several
# passes over the row (one slot per CTA); the head stays the same launch.
@pytest.mark.parametrize("slots", [5, 8, 17, 50])
@pytest.mark.parametrize("width,actions", [(64, 1), (1024, 20), (1032, 32)])
def test_head_tail_many_rows(slots, width, actions):
    batch = 2 * torch.cuda.get_device_properties(0).multi_processor_count // slots + 1
    cfg = synth.ExpertConfig(layers=1, width=width, n_q_heads=2, n_kv_heads=1, head_dim=64, mlp_dim=64, slots=slots,
                             action_dim=actions, prefix=9, fop_tokens=2, batch=batch, dtype="bf16")
    case = Case(cfg)
    s = gpu_session(case)
    for _ in range(2):
        check_step(case, s, robots=[0, batch // 2, batch - 1], label=f"{batch * slots} rows")
    few = gpu_session(Case(cfg, batch=1))
    check_step(Case(cfg, batch=1), few)
    assert s.kernel_count() == few.kernel_count()
    s.close()
    few.close()


# Token counts where a step's projections exchange fp32 shares or sum two halves
# (QKV at 129 to 192 tokens; O and down at 513 to 576 and at 577 to 1152), and
# attentions whose few splits merge in fp32 through L2 or whose one prefix chunk
# is not split.
@pytest.mark.parametrize("batch,slots,heads,kv,hd,prefix", [(2, 50, 8, 1, 256, 300), (11, 50, 8, 1, 256, 100),
                                                            (16, 50, 8, 1, 256, 64), (19, 8, 8, 2, 80, 384),
                                                            (2, 30, 16, 4, 64, 2048), (3, 30, 16, 4, 64, 64)])
def test_exchange_in_fp32(batch, slots, heads, kv, hd, prefix):
    cfg = synth.ExpertConfig(layers=1, width=1024, n_q_heads=heads, n_kv_heads=kv, head_dim=hd, mlp_dim=4096,
                             slots=slots, action_dim=7, prefix=prefix, fop_tokens=16, batch=batch, dtype="bf16")
    case = Case(cfg)
    s = gpu_session(case)
    check_step(case, s, robots=[0, batch - 1], label=f"{batch * slots} tokens")
    s.close()
