"""CPU checks of which host tensors the banded host steps hand to the native
call: exactly those for which writing through their data pointer is what
torch's copies would do."""
import pytest

torch = pytest.importorskip("torch")


@pytest.fixture
def run(monkeypatch):
    from paper_2205_07572_gb300 import af
    from paper_2205_07572_gb300.uniform import UniformRun
    calls = []
    monkeypatch.setattr(af, "step_host_bands", lambda *a: calls.append(a))
    r = UniformRun.__new__(UniformRun)
    r.cfg, r.tiling, r.dt, r.dx, r.dy, r.t, r.freg = None, 0, 0.5, 1.0, 1.0, 0.0, None
    r.npatch, r.words = 1, 6
    r.a = r.b = torch.zeros((1, 6))
    r._streams, r._bands_c, r._mark = (None, None, None), (), torch.zeros(1)
    return lambda host: (r._step_host_native(host, 6, None, None), len(calls), r)


def test_a_plain_tensor_is_written_natively_and_its_version_counted(run):
    host = torch.ones((1, 6))
    v = host._version
    done, calls, r = run(host)
    assert done and calls == 1 and r.t == 0.5 and host._version > v
    # autograd sees the write: a graph that saved the old values refuses to use them
    w = torch.ones((1, 6), requires_grad=True)
    out = (w * host).sum()
    run(host)
    with pytest.raises(RuntimeError, match="modified by an inplace operation"):
        out.backward()


def _inference():
    with torch.inference_mode():
        return torch.ones((1, 6))


class _Sub(torch.Tensor):
    pass


@pytest.mark.parametrize("host", [
    torch.ones((1, 6), requires_grad=True),
    torch.nn.Parameter(torch.ones((1, 6))),
    torch.ones((1, 6)).as_subclass(_Sub),
    torch._neg_view(torch.ones((1, 6))),
    _inference(),
    torch.ones((1, 6), dtype=torch.float64),
    torch.ones((1, 12))[:, ::2],
    torch.ones(6), torch.ones((1, 6)).numpy(),
], ids=["requires_grad", "parameter", "subclass", "negated", "inference", "double", "strided", "flat", "numpy"])
def test_other_forms_go_through_torchs_copies(run, host):
    done, calls, r = run(host)
    assert not done and calls == 0 and r.t == 0.0 and not r._mark.requires_grad


def test_a_parameter_without_gradient_is_written_natively(run):
    done, calls, _ = run(torch.nn.Parameter(torch.ones((1, 6)), requires_grad=False))
    assert done and calls == 1


def test_inference_mode_writes_its_own_tensors(run):
    with torch.inference_mode():
        done, calls, _ = run(torch.ones((1, 6)))
    assert done and calls == 1
