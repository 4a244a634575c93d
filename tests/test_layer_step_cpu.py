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


def gpu(*shape, dtype=torch.float32):
    return torch.zeros(shape, dtype=dtype).as_subclass(OnGpu)


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
