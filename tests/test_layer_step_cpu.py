"""What a layer-step hands to the library, checked on the host: the call's fields for given tensors,
hyper-parameters and layers, and the arguments that are refused.  Nothing is launched: the library
entry is replaced by one that records its arguments, and the tensors only claim to be on a GPU."""
import ctypes

import numpy as np
import pytest
import torch

import paper_2406_17660_b200 as grass
from paper_2406_17660_b200 import binding as B


class OnGpu(torch.Tensor):
    """A host tensor that answers as a CUDA tensor does."""
    is_cuda = True

    def __deepcopy__(self, memo):
        return memo.setdefault(id(self), self.clone().as_subclass(OnGpu))


def gpu(*shape, dtype=torch.float32):
    return torch.zeros(shape, dtype=dtype).as_subclass(OnGpu)


LAUNCHING = ("grass_grad_row_norms", "grass_select", "grass_project_grad", "grass_project_grad_batched",
             "grass_adam_scatter_batched")


@pytest.fixture
def calls(monkeypatch):
    """The (entry, grass_step_t fields, grass_refresh_t fields) of every call that would be launched."""
    seen = []

    def fields(ref):
        s = ref._obj
        return {n: (list(v) if isinstance(v, ctypes.Array) else v)
                for n, v in ((f[0], getattr(s, f[0])) for f in s._fields_)}

    def layer_step(step, stream):
        seen.append(("step", fields(step), None))
        return 0

    def refresh_step(step, refresh, stream):
        seen.append(("refresh", fields(step), fields(refresh)))
        return 0

    real = B.load_library()

    class Library:
        grass_layer_step = staticmethod(layer_step)
        grass_refresh_step = staticmethod(refresh_step)

        def __getattr__(self, name):
            if name in LAUNCHING:
                return lambda *args: seen.append((name, args, None)) or 0
            return getattr(real, name)

    library = Library()
    monkeypatch.setattr(B, "load_library", lambda: library)
    monkeypatch.setattr(B, "_stream", lambda: 0)
    return seen


T, M, N, R = 64, 48, 40, 8
HYPER = (1e-3, 0.9, 0.999, 1e-8)


def buffers(r=R, m=M, n=N):
    return dict(idx=gpu(r, dtype=torch.int32), rho=gpu(r), Gc=gpu(r, n), M=gpu(r, n), V=gpu(r, n),
                U=gpu(r, n), W=gpu(m, n, dtype=torch.bfloat16))


def test_a_hyper_parameter_changed_in_place_reaches_the_next_call(calls):
    """lr and alpha may be 0-d arrays that a schedule writes to: the call reads their value, not who they are."""
    call = B.LayerStepCall()
    call.state(0, **buffers())
    call.inputs(0, gpu(T, M, dtype=torch.bfloat16), gpu(T, N, dtype=torch.bfloat16))
    lr, alpha = np.array(1e-3), torch.tensor(0.25, dtype=torch.float64)
    for step in (1, 2):
        call.launch(1, None, lr, 0.9, 0.999, 1e-8, step, alpha)
        lr *= 0.5
        alpha *= 2
    assert [c[1]["lr"] for c in calls] == [1e-3, 5e-4]
    assert [c[1]["alpha"] for c in calls] == [0.25, 0.5]


@pytest.mark.parametrize("name,bad,error", [
    ("rho", torch.zeros(R), TypeError),                          # host memory
    ("rho", gpu(R, dtype=torch.float64), TypeError),
    ("rho", gpu(R, dtype=torch.bfloat16), TypeError),
    ("rho", gpu(R - 1), ValueError),
    ("rho", gpu(2 * R)[::2], ValueError),
    ("idx", torch.zeros(R, dtype=torch.int32), TypeError),
    ("idx", gpu(R, dtype=torch.int64), TypeError),
    ("idx", gpu(R - 1, dtype=torch.int32), ValueError),
    ("idx", gpu(2 * R, dtype=torch.int32)[::2], ValueError),
    ("U", torch.zeros(R, N), TypeError),
    ("U", gpu(R, N, dtype=torch.float64), TypeError),
    ("U", gpu(R - 1, N), ValueError),
    ("U", gpu(R, N - 1), ValueError),
    ("U", gpu(R, N + 8)[:, :N], ValueError),                     # not M's pitch
    ("M", gpu(R, N + 1), ValueError), ("V", gpu(R - 1, N), ValueError), ("Gc", gpu(R, N, dtype=torch.float64), TypeError),
    ("W", gpu(M, N, dtype=torch.float16), TypeError), ("W", gpu(M, N + 1), ValueError),
], ids=lambda v: v if isinstance(v, str) else "")
def test_a_layers_buffers_are_checked_before_a_call_points_at_them(calls, name, bad, error):
    with pytest.raises(error):
        B.LayerStepCall().state(0, **dict(buffers(), **{name: bad}))


def test_what_a_layer_may_leave_out_or_have_to_spare(calls):
    call = B.LayerStepCall()
    call.state(0, **dict(buffers(), U=None, rho=None))
    assert call.args.U[0] is None and call.args.rho[0] is None
    longer = dict(buffers(), idx=gpu(R + 3, dtype=torch.int32), rho=gpu(R + 3))
    call.state(0, **longer)
    assert call.args.r == R and call.args.rho[0] == longer["rho"].data_ptr()


def layer(m=M, n=N, r=R, tokens=T, K=2, t=0, **kw):
    W = gpu(m, n, dtype=torch.bfloat16)
    ws = grass.step.GrassWorkspace([(m, n)], tokens, r, torch.bfloat16, grass.SEL_TOPR, device="cpu")
    ws.norms = ws.norms.as_subclass(OnGpu)
    kw = dict(dict(alpha=0.25, lr=1e-3), **kw)
    l = grass.GrassLayer(W, r, grass.SEL_TOPR, K, workspace=ws, **kw)
    for name in ("idx", "rho", "Gc", "M", "V", "U"):
        setattr(l, name, getattr(l, name).as_subclass(OnGpu))
    l.t = t
    return l


def bf16(count, *shape):
    return [gpu(*shape, dtype=torch.bfloat16) for _ in range(count)]


def test_a_group_steps_the_tensors_that_its_layers_have_now(calls):
    """A layer whose state or weights were replaced (a checkpoint loaded) after the group was made."""
    group = grass.step.GrassLayerGroup([layer(t=1), layer(t=1)], T, device="cpu")
    group.step(bf16(2, T, M), bf16(2, T, N))
    second = group.layers[1]
    for name in ("idx", "rho", "Gc", "M", "V", "U", "W"):
        setattr(second, name, getattr(second, name).clone().as_subclass(OnGpu))
        second.t = group.layers[0].t = 1
        group.step(bf16(2, T, M), bf16(2, T, N))
        assert calls[-1][1][name][1] == getattr(second, name).data_ptr(), name
        assert calls[-1][1][name][0] == getattr(group.layers[0], name).data_ptr()


def test_a_copied_group_steps_its_own_layers(calls):
    import copy
    group = grass.step.GrassLayerGroup([layer(t=1), layer(t=1)], T, device="cpu")
    other = copy.deepcopy(group)
    other.step(bf16(2, T, M), bf16(2, T, N))
    for g in range(2):
        assert calls[-1][1]["W"][g] == other.layers[g].W.data_ptr() != group.layers[g].W.data_ptr()
