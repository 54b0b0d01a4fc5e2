"""AisStep as an object, without a GPU: the library's step entry is replaced by one that notes what it is given."""

import ctypes

import pytest
import torch

T, D, V, P, G = 96, 256, 1024, 2, 3
TENSORS = ("workspace", "qH", "qW", "sH", "sW", "lp_train", "lse_train", "lp_roll", "lse_roll", "rho", "w_tilde", "adv", "n_valid_seq",
           "loss", "diag", "status", "dH")


class Recorder:
    """Stands in for the loaded library: every ais_step call's argument struct, by field name."""

    def __init__(self, real, binding):
        self.real, self.binding, self.calls = real, binding, []

    def __getattr__(self, name):
        return getattr(self.real, name)

    def ais_step(self, shape, params, args, stages, stream):
        a = ctypes.cast(args, ctypes.POINTER(self.binding.StepArgs)).contents
        self.calls.append({n: getattr(a, n) for n, _ in self.binding.StepArgs._fields_})
        return 0


@pytest.fixture
def recorder(monkeypatch):
    from paper_2605_13907_b200 import binding
    r = Recorder(binding.lib(), binding)
    monkeypatch.setattr(binding, "lib", lambda: r)
    monkeypatch.setattr(binding, "_require_cuda", lambda *t: None)
    monkeypatch.setattr(binding, "_stream", lambda t: 0)
    return r


def _inputs():
    return dict(H=torch.zeros(T, D, dtype=torch.bfloat16), W=torch.zeros(V, D, dtype=torch.bfloat16), tokens=torch.zeros(T, dtype=torch.int32),
                mask=torch.ones(T, dtype=torch.uint8))


def _step_inputs():
    return dict(_inputs(), seq_offsets=torch.zeros(P * G + 1, dtype=torch.int32), rewards=torch.zeros(P * G))


def _step():
    from paper_2605_13907_b200 import AisStep
    return AisStep(T, D, V, P, G, 128, device="cpu")


@pytest.mark.parametrize("how", ["data", "set_", "resize_", "assign"])
@pytest.mark.parametrize("name", TENSORS)
def test_a_buffer_that_moved_is_used_where_it_is(recorder, name, how):
    """Each way to give a step's tensor other storage between two calls."""
    step, x = _step(), _step_inputs()
    step.step(**x)
    t = getattr(step, name)
    other = torch.zeros_like(t)
    if how == "data":
        t.data = other
    elif how == "set_":
        t.set_(other)
    elif how == "resize_":
        t.resize_(4 * max(t.numel(), 1 << 20)).resize_(other.shape)
    else:
        setattr(step, name, other)
    step.step(**x)
    field = "dev_status" if name == "status" else name
    assert recorder.calls[1][field] == getattr(step, name).data_ptr()
    if how != "resize_":
        assert recorder.calls[1][field] != recorder.calls[0][field]


def test_a_workspace_that_shrank_in_place_is_passed_with_its_size(recorder):
    step, x = _step(), _step_inputs()
    step.step(**x)
    step.workspace.resize_(step.workspace.numel() - 4096)
    step.step(**x)
    assert recorder.calls[1]["workspace_bytes"] == recorder.calls[0]["workspace_bytes"] - 4096 == step.workspace.numel()


def test_strides_of_the_scales_are_read_at_every_call(recorder):
    step, x = _step(), _step_inputs()
    step.step(**x)
    wide = torch.zeros(step.sW.shape[0], step.sW.shape[1] + 64)
    step.sW.set_(wide)
    step.step(**x)
    assert recorder.calls[1]["ldsW"] == wide.stride(0)


@pytest.mark.parametrize("how", ["copy", "deepcopy", "pickle"])
def test_a_step_that_has_run_can_be_copied(recorder, how):
    """A copy shares the tensors, a deep copy and a pickled one have their own."""
    import copy
    import pickle
    step, x = _step(), _step_inputs()
    step.step(**x)
    other = {"copy": copy.copy, "deepcopy": copy.deepcopy, "pickle": lambda s: pickle.loads(pickle.dumps(s))}[how](step)
    other.step(**x)
    for name in ("workspace", "lp_train", "dH"):
        assert recorder.calls[1][name] == getattr(other, name).data_ptr()
        assert (recorder.calls[1][name] == recorder.calls[0][name]) == (how == "copy")


@pytest.mark.parametrize("where", ["subclass", "instance"])
@pytest.mark.parametrize("name", ["quantize_weights", "forward", "diagnose", "backward"])
def test_a_stage_that_was_replaced_is_called(recorder, monkeypatch, name, where):
    """step() is made of the four stages: one that a subclass or a program puts its own in place of is run."""
    from paper_2605_13907_b200 import binding
    for f in ("quantize_fp8", "logprob_fwd", "diagnostics", "loss_bwd"):
        monkeypatch.setattr(binding, f, lambda *a, **k: None)
    seen = []
    if where == "subclass":
        cls = type("Own", (binding.AisStep,), {name: lambda self, *a, **k: seen.append(name)})
        step = cls(T, D, V, P, G, 128, device="cpu")
    else:
        step = _step()
        setattr(step, name, lambda *a, **k: seen.append(name))
    step.step(**_step_inputs())
    assert seen == [name]


def test_replaced_weight_quantiser_is_called_by_forward(recorder, monkeypatch):
    from paper_2605_13907_b200 import binding
    for f in ("quantize_fp8", "logprob_fwd"):
        monkeypatch.setattr(binding, f, lambda *a, **k: None)
    step, seen = _step(), []
    step.quantize_weights = seen.append
    x = _inputs()
    step.forward(**x)
    assert seen == [x["W"]]


def test_two_threads_calls_do_not_share_their_arguments(recorder):
    """A call that is still inside the library (which runs without the interpreter's lock) keeps its own inputs when another
    thread calls the same step."""
    import threading
    step, inside, go = _step(), threading.Event(), threading.Event()
    x, y = _step_inputs(), _step_inputs()
    note = recorder.ais_step

    def slow(shape, params, args, stages, stream):
        if threading.current_thread() is not threading.main_thread():
            inside.set()
            assert go.wait(20)
        return note(shape, params, args, stages, stream)

    recorder.ais_step = slow
    step.step(**_step_inputs())
    t = threading.Thread(target=lambda: step.step(**x))
    t.start()
    assert inside.wait(20)
    step.step(**y)
    go.set()
    t.join()
    assert [c["H"] for c in recorder.calls[1:]] == [y["H"].data_ptr(), x["H"].data_ptr()]
