"""The step driver's host side (buffers, views, what it hands to the library), on the CPU with the library's calls recorded."""
import pytest
import torch

import paper_2609_17380_b200 as det
from paper_2609_17380_b200 import step as dstep

HOST = ("det_accum", "det_adamw_desc", "det_grad_accum_nbufs")


@pytest.fixture
def calls(monkeypatch):
    """(name, arguments) of every library call that would launch something."""
    log = []
    for name in dir(det):
        if name.startswith("det_") and not name.endswith("ws_bytes") and name not in HOST:
            monkeypatch.setattr(det, name, lambda *a, _name=name, **k: log.append((_name, a)))
    return log


@pytest.fixture
def counted_losses(calls, monkeypatch):
    """The losses of successive forward passes are 1, 2, ..."""
    n = [0.0]

    def xent(logits, target, rows, V, z, loss_row, lse, loss_mean, *rest):
        n[0] += 1.0
        loss_mean.fill_(n[0])

    monkeypatch.setattr(det, "det_xent_fwd", xent)
    monkeypatch.setattr(torch.cuda.nvtx, "range_push", lambda *a: None)
    monkeypatch.setattr(torch.cuda.nvtx, "range_pop", lambda *a: None)


def _replay(**kw):
    cfg = dict(n_layers=2, d_model=256, n_heads=2, ffn=256, vocab=512, seq=64, micro_batch=2, mesh=(1, 2, 1))
    cfg.update(kw)
    return dstep.Replay(dstep.ModelConfig(**cfg), device="cpu")


# tokens of a micro-batch: [rows, sequence + 1] of the configuration, or any rows whose tokens come to the same number
@pytest.mark.parametrize("shape", [(2, 65), (1, 129), (4, 33), (128, 2)])
def test_tokens_accepted(calls, shape):
    r = _replay()
    t = torch.arange(shape[0] * shape[1], dtype=torch.int32).reshape(shape)
    r.forward(t)
    assert torch.equal(r.tok, t[:, :-1].reshape(-1)) and torch.equal(r.lab, t[:, 1:].reshape(-1))


# too few or too many are refused, one row for all sequences and one token for all positions among them
@pytest.mark.parametrize("shape", [(1, 65), (2, 2), (2, 64), (3, 65), (2, 1)])
def test_tokens_refused(calls, shape):
    r = _replay()
    with pytest.raises(RuntimeError):
        r.forward(torch.zeros(shape, dtype=torch.int32))


# loss_mean is one buffer: who holds it sees the loss of the latest forward pass, and a forward pass after a step leaves what
# the step reports alone
def test_loss_buffer_stays(calls, counted_losses):
    r = _replay()
    held = r.loss_mean
    tokens = torch.zeros((2, 2, 65), dtype=torch.int32)
    assert r.step(tokens)["losses"] == [1.0, 2.0]
    assert held is r.loss_mean and held.item() == 2.0
    r.forward(tokens[0])
    assert held.item() == 3.0 and r._losses.tolist() == [1.0, 2.0]


# a buffer of the state replaced, or given other memory, between two calls: the library gets the memory that is there now
@pytest.mark.parametrize("swap", ["object", "memory"])
def test_replaced_buffers_are_used(calls, swap):
    r = _replay()
    t = torch.zeros((2, 65), dtype=torch.int32)

    def passes():
        del calls[:]
        r.prepare_weights()
        r.forward(t, calibrate=True)
        r.forward(t)
        r.backward()
        r.optimizer()

    def touched():
        return {a.data_ptr() for _, args in calls for x in args for a in (x if isinstance(x, list) else [x]) if torch.is_tensor(a)}

    passes()
    names, old = ("sx", "pbf", "m", "v", "gmb"), {}
    for n in names:
        old[n] = getattr(r, n).detach()[:]                  # keeps the old memory, so that no new buffer can be at its address
        if swap == "object":
            setattr(r, n, getattr(r, n).clone())
        else:
            getattr(r, n).data = getattr(r, n).clone()
    passes()
    for n in names:
        lo = old[n].data_ptr()
        stale = [p for p in touched() if lo <= p < lo + old[n].numel() * old[n].element_size()]
        assert not stale, n
    steps = {r.sx.data_ptr() + 4 * i for i in range(8)}
    assert steps <= touched()


# the scalars and roots that a step reports are those of the tensors the library was given, also where one of them was replaced
def test_replaced_report_is_read(calls, counted_losses, monkeypatch):
    r = _replay()
    tokens = torch.zeros((2, 2, 65), dtype=torch.int32)
    r.status, r.norm, r.coef = torch.tensor([4], dtype=torch.int32), torch.tensor([0.5]), torch.tensor([0.25])
    monkeypatch.setattr(det, "det_tensor_hash_batch", lambda ts, roots, ws: roots.copy_(torch.arange(roots.numel()) % 251))
    for moved in (False, True):
        if moved:
            r.roots = torch.zeros_like(r.roots)
        res = r.step(tokens)
        assert (res["status"], res["grad_norm"], res["coef"]) == (4, 0.5, 0.25)
        assert res["hashes"]["embed"] == bytes(range(32)).hex()
