"""RollingSession's step inputs, without a GPU: CPU tensors stand in for the
device's, and the one-launch copy is replaced by one that reads every value
before it writes any, in the reverse order -- as good an order as any for
arrays that may not overlap."""
import ctypes

import pytest

torch = pytest.importorskip("torch")


@pytest.fixture
def session(monkeypatch):
    from paper_2609_34170_gb300 import session as mod
    s = object.__new__(mod.RollingSession)
    s.torch, s.device, s.dtype, s.handle = torch, torch.device("cpu"), torch.float32, None
    s.slot_times, s.delta = torch.zeros(6), torch.zeros(4)
    s.obs, s.state = torch.zeros(4, 3, 8), torch.zeros(4, 2)
    s.launches = 0

    def copy(handle, n, dst, src, nbytes, stream=None):
        s.launches += 1
        assert all(dst[i] and src[i] for i in range(n))
        data = [ctypes.string_at(src[i], nbytes[i]) for i in range(n)]
        for i in reversed(range(n)):
            ctypes.memmove(dst[i], data[i], nbytes[i])

    monkeypatch.setattr(mod.B, "ravel_copy_inputs", copy)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda device=None: None)
    return s


def _put(s, times, obs, delta, state):
    s._put(s._times(times), (s.obs, obs), (s.delta, delta), (s.state, state))


def test_plain_tensors_take_one_launch(session):
    t, o, d, a = torch.rand(6), torch.rand(4, 3, 8), torch.rand(4), torch.rand(4, 2)
    _put(session, t, o, d, a)
    assert session.launches == 1
    for got, want in ((session.slot_times, t), (session.obs, o), (session.delta, d), (session.state, a)):
        assert torch.equal(got, want)
    _put(session, session.slot_times, o, session.delta, a)   # a value that is its own input
    assert torch.equal(session.slot_times, t) and torch.equal(session.delta, d)


def test_values_that_are_other_inputs_buffers_are_copied_in_order(session):
    t, o, a = torch.rand(6), torch.rand(4, 3, 8), torch.rand(4, 2)
    _put(session, t, o, session.slot_times[:4], a)            # ages from the slot times of this very step
    assert torch.equal(session.delta, t[:4])
    t2, o2, d = torch.rand(6), torch.rand(4, 3, 8), torch.rand(4)
    _put(session, t2, o2, d, session.obs[:, 0, :2].contiguous())
    assert torch.equal(session.state, o[:, 0, :2])            # (a copy made before the call)
    _put(session, t2, o, d, session.obs.view(-1)[:8].view(4, 2))
    assert torch.equal(session.state, o.view(-1)[:8].view(4, 2))
    with pytest.raises(RuntimeError):                         # part of its own input: the copy refuses
        _put(session, session.slot_times[2:5], o, d, a)
    _put(session, session.obs.view(-1)[3:9], o2, d, a)        # the tokens of the step before
    assert torch.equal(session.slot_times, o.view(-1)[3:9])


def test_fewer_or_no_slot_times_keep_the_rest(session):
    _put(session, torch.arange(6.0), torch.rand(4, 3, 8), torch.rand(4), torch.rand(4, 2))
    _put(session, torch.empty(0), torch.rand(4, 3, 8), torch.rand(4), torch.rand(4, 2))
    _put(session, torch.tensor([9.0, 8.0]), torch.rand(4, 3, 8), torch.rand(4), torch.rand(4, 2))
    assert session.slot_times.tolist() == [9.0, 8.0, 2.0, 3.0, 4.0, 5.0]


def test_inputs_before_one_that_does_not_fit_are_taken(session):
    t = torch.rand(6)
    with pytest.raises(RuntimeError):
        _put(session, t, torch.rand(4, 3, 9), torch.rand(4), torch.rand(4, 2))
    assert torch.equal(session.slot_times, t) and not session.delta.any()
