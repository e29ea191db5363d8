"""Per-robot context swaps through the C ABI (ravel_set_context_robots).

In the paper every robot's VLM context is refreshed asynchronously, whenever
its own VLM pass completes (Method, "Asynchronous Context Updates"): robots
then run with contexts of different ages and lengths.  The library keeps a
double-buffered context per robot; a swap for some robots leaves the others'
contexts untouched.  Each step is held to the step tolerances of the oracle
run with every robot's own context and prefix length.
"""
import numpy as np
import pytest

import synth
from oracle import expert
from tests._harness import TOL, Case, gpu_session, rel_l2

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2609_34170_gb300 import build, load
    build.build()
    load()


def _cfg(dtype):
    return synth.ExpertConfig(layers=2, width=192, n_q_heads=6, n_kv_heads=2, head_dim=40, mlp_dim=320, slots=7,
                              action_dim=5, prefix=45, fop_tokens=3, batch=3, dtype=dtype)


class _Contexts:
    """The oracle's view: every robot's current K/V rows and prefix length."""

    def __init__(self, cfg, k, v, P):
        L, B, Hkv, _, hd = k.shape
        self.k = np.zeros((L, B, Hkv, cfg.prefix, hd), k.dtype)
        self.v = np.zeros_like(self.k)
        self.P = np.zeros(B, np.int64)
        self.install(list(range(B)), k, v, P)

    def install(self, robots, k, v, P):
        for i, b in enumerate(robots):
            self.k[:, b] = 0
            self.v[:, b] = 0
            self.k[:, b, :, :P] = k[:, i, :, :P]
            self.v[:, b, :, :P] = v[:, i, :, :P]
            self.P[b] = P


def _step_and_check(case, s, ctx, label):
    buf0 = s.buffer.cpu().numpy().copy()
    cnt0 = np.asarray(s.counters(), np.uint64)
    s.step(case.t, case.fop, case.delta, want_velocity=True)
    torch.cuda.synchronize()
    rel_o, new_o, cnt_o, vel_o = expert.roll_step(case.cfg, case.W, buf0, case.t, ctx.k, ctx.v, ctx.P, case.fop,
                                                  case.delta, case.seeds, cnt0)
    tol_a, tol_v = TOL[case.cfg.dtype]
    err_a = float(np.max(np.abs(s.released.cpu().numpy() - rel_o)))
    err_v = rel_l2(s.velocity.cpu().numpy(), vel_o)
    assert err_a <= tol_a, f"{label}: released max-abs {err_a:.3e}"
    assert err_v <= tol_v, f"{label}: velocity rel-L2 {err_v:.3e}"
    np.testing.assert_array_equal(s.counters(), cnt_o)
    return vel_o


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
def test_some_robots_swap_while_the_others_keep_their_context(dtype):
    from paper_2609_34170_gb300 import RollingSession
    cfg = _cfg(dtype)
    case = Case(cfg)
    s = RollingSession(cfg, case.W, 0, cfg.batch, cfg.prefix)
    s.reset(case.seeds)
    s.set_context(case.k, case.v, case.P)
    ctx = _Contexts(cfg, case.k, case.v, case.P)
    _step_and_check(case, s, ctx, "all robots, context A")
    # robots 0 and 2 receive context B (shorter), robot 1 keeps A
    kb, vb = synth.make_context(cfg, 3000, 2, 30)
    s.set_context_robots([2, 0], kb, vb, 30)
    ctx.install([2, 0], kb, vb, 30)
    _step_and_check(case, s, ctx, "robots 0, 2 on B")
    # robot 1 receives context C (much shorter); 0 and 2 keep B
    kc, vc = synth.make_context(cfg, 4000, 1, 12)
    s.set_context_robots([1], kc, vc, 12)
    ctx.install([1], kc, vc, 12)
    _step_and_check(case, s, ctx, "robot 1 on C")
    # and a step with no swap reuses every robot's context
    _step_and_check(case, s, ctx, "no swap")
    s.close()


def test_per_robot_swap_rules():
    from paper_2609_34170_gb300 import RavelError, RollingSession
    cfg = _cfg("bf16")
    case = Case(cfg)
    s = RollingSession(cfg, case.W, 0, cfg.batch, cfg.prefix)
    s.reset(case.seeds)
    # robots 0 and 1 only: a step needs every robot's context
    kb, vb = synth.make_context(cfg, 3000, 2, 20)
    s.set_context_robots([0, 1], kb, vb, 20)
    with pytest.raises(RavelError, match="ENOCONTEXT"):
        s.step(case.t, case.fop, case.delta)
    kc, vc = synth.make_context(cfg, 4000, 1, 20)
    s.set_context_robots([2], kc, vc, 20)
    # robot 0's swap is still pending: a second one for it is refused
    with pytest.raises(RavelError, match="EBUSY"):
        s.set_context_robots([0], kc, vc, 20)
    with pytest.raises(RavelError, match="EINVAL"):
        s.set_context_robots([1, 1], kb, vb, 20)
    with pytest.raises(RavelError, match="EINVAL"):
        s.set_context_robots([3], kc, vc, 20)
    ctx = _Contexts(cfg, case.k, case.v, case.P)   # replaced below
    ctx.install([0, 1], kb, vb, 20)
    ctx.install([2], kc, vc, 20)
    _step_and_check(case, s, ctx, "contexts assembled from two calls")
    s.close()


# The session's step inputs: plain CUDA tensors go in one launch, everything else
# one by one; all forms give the same step, and what cannot fill an input is
# refused as before.
@pytest.mark.parametrize("fop", [0, 3])
def test_step_inputs_in_every_form(fop):
    cfg = synth.ExpertConfig(layers=1, width=72, n_q_heads=2, n_kv_heads=1, head_dim=24, mlp_dim=64, slots=5,
                             action_dim=3, prefix=9, fop_tokens=fop, batch=3, dtype="bf16")
    case = Case(cfg)
    outs = []
    dev = lambda a, dt=torch.float32: torch.from_numpy(np.ascontiguousarray(a)).to("cuda", dt)  # noqa: E731
    t, d, z = dev(case.t), dev(case.delta), dev(case.fop, torch.bfloat16)
    odd = torch.zeros(t.numel() + 1, device="cuda")[1:]   # 4-byte aligned only
    odd.copy_(t)
    forms = [(case.t, case.fop, case.delta), (t, z, d), (odd, z, d), (t.reshape(1, -1), z.float(), d.double()),
             (t, z.transpose(0, 1).contiguous().transpose(0, 1), d), (t, z, case.delta)]
    for tt, zz, dd in forms:
        s = gpu_session(case)
        s.step(tt, zz, dd, want_velocity=True)
        outs.append((s.released.clone(), s.velocity.clone()))
        with pytest.raises(RuntimeError):
            s.step(t, z, d.reshape(-1, 1))
        with pytest.raises(RuntimeError):
            s.step(torch.cat([t, t]), z, d)
        s.close()
    for r, v in outs[1:]:
        assert torch.equal(r, outs[0][0]) and torch.equal(v, outs[0][1])


def _raw_step(case, s, bad=None):
    """One step from a fresh rollout: released actions and velocity.  Robot
    `bad`'s actions and observation are not numbers."""
    s.reset(case.seeds)
    fop = case.fop.copy()
    if bad is not None:
        s.buffer[bad] = float("nan")
        fop[bad] = np.nan
    s.step(case.t, fop, case.delta, want_velocity=True)
    torch.cuda.synchronize()
    return s.released.cpu().numpy(), s.velocity.cpu().numpy()


# head dims with one and four 64-wide blocks; slots + FOP tokens that end inside
# a group of 16 keys; one robot group whose keys are split and one whose are not
@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
@pytest.mark.parametrize("heads,kv,hd", [(6, 2, 40), (4, 1, 64), (4, 1, 256)])
@pytest.mark.parametrize("B,slots", [(2, 7), (48, 50)])
def test_a_robots_bad_values_stay_its_own(dtype, heads, kv, hd, B, slots):
    # keys of another robot have probability 0, but 0 x NaN is NaN
    cfg = synth.ExpertConfig(layers=2, width=192, n_q_heads=heads, n_kv_heads=kv, head_dim=hd, mlp_dim=320,
                             slots=slots, action_dim=5, prefix=45, fop_tokens=3, batch=B, dtype=dtype)
    case = Case(cfg)
    s = gpu_session(case)
    clean, got = _raw_step(case, s), _raw_step(case, s, bad=1)
    others = [b for b in range(B) if b != 1]
    for c, g in zip(clean, got):
        np.testing.assert_array_equal(g[others], c[others])
        assert np.isnan(g[1]).all()   # and the robot itself is told
    s.close()


@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
@pytest.mark.parametrize("P", [1, 18, 32])
def test_rows_of_an_earlier_longer_context_are_never_used(dtype, P):
    cfg = _cfg(dtype)
    case = Case(cfg, prefix_len=P)
    s = gpu_session(case)
    want = _raw_step(case, s)
    s.close()
    k, v = synth.make_context(cfg, 5000, cfg.batch, cfg.prefix)
    v[..., P:, :] = np.nan
    s = gpu_session(case)
    for c in ((k, v, cfg.prefix), (k, v, cfg.prefix), (case.k, case.v, P)):   # the slots alternate
        s.step(case.t, case.fop, case.delta)
        s.set_context(*c)
    got = _raw_step(case, s)
    for c, g in zip(want, got):
        np.testing.assert_array_equal(g, c)
    s.close()
