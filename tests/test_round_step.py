"""What EARound.step hands to the library, without a GPU: the C functions are replaced by ones that read each
gradient when it is handed over, as a launch on the stream would."""
import ctypes

import pytest
import torch

import paper_2205_14473_gb300 as ea
from paper_2205_14473_gb300 import workloads as W

D, N = 8, 4


@pytest.fixture
def rnd(monkeypatch):
    r = ea.EARound.__new__(ea.EARound)
    r.cfg = ea.EAConfig(d=D, n=N, qw=W.sign_q(0), qs=W.sign_q(0), alpha=1e-3)
    r.h = 0  # no handle to destroy
    r.log = []

    def read(p):
        return list((ctypes.c_float * D).from_address(p))

    monkeypatch.setattr(ea, "ea_worker_compress", lambda h, i, p: r.log.append((i, read(p))))
    monkeypatch.setattr(ea, "ea_server_step", lambda h: r.log.append("server"))
    monkeypatch.setattr(ea, "ea_worker_apply", lambda h, p: r.log.append("apply"))

    def round_step(h, ps, x):
        r.log += [(i, read(p)) for i, p in enumerate(ps)] + ["server", "apply", "one call"]

    monkeypatch.setattr(ea, "ea_round_step", round_step)
    return r


def _want():
    return [(i, [float(i)] * D) for i in range(N)] + ["server", "apply"]


class _OneBuffer:
    """Worker i's gradient, formed when it is asked for, in the one buffer there is."""

    def __init__(self):
        self.buf, self.asked = torch.empty(D), []

    def __getitem__(self, i):
        self.asked.append(i)
        return self.buf.fill_(float(i))


def test_gradients_formed_in_one_buffer(rnd):
    gs = _OneBuffer()
    rnd.step(gs, torch.zeros(D))
    assert rnd.log == _want()
    assert gs.asked == list(range(N))  # each once, after the worker before it was handed over


def test_a_list_subclass_may_do_the_same(rnd):
    class Lazy(list):
        buf = torch.empty(D)

        def __getitem__(self, i):
            return self.buf.fill_(float(i))

    rnd.step(Lazy([None] * N), torch.zeros(D))
    assert rnd.log == _want()


@pytest.mark.parametrize("kind", [list, tuple, torch.stack])
def test_tensors_at_hand_share_one_call(rnd, kind):
    rnd.step(kind([torch.full((D,), float(i)) for i in range(N)]), torch.zeros(D))
    assert rnd.log == _want() + ["one call"]


@pytest.mark.parametrize("bad", ["strided", "short", "integer", "missing", "x"])
def test_what_is_not_accepted_fails_where_its_own_call_does(rnd, bad):
    gs, x = [torch.full((D,), float(i)) for i in range(N)], torch.zeros(D)
    if bad == "missing":
        del gs[2:]
    elif bad == "x":
        x = torch.zeros(2 * D)[::2]
    else:
        gs[2] = {"strided": torch.zeros(2 * D)[::2], "short": torch.zeros(D - 1),
                 "integer": torch.zeros(D, dtype=torch.int32)}[bad]
    with pytest.raises((AssertionError, IndexError)):
        rnd.step(gs, x)
    assert rnd.log == (_want()[:-1] if bad == "x" else _want()[:2])
