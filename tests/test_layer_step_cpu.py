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
             "grass_adam_scatter_batched", "grass_subspace_adam", "grass_scatter_update", "grass_scatter_update_cols")


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


def layer(m=M, n=N, r=R, tokens=T, K=2, t=0, cls=grass.GrassLayer, **kw):
    W = gpu(m, n, dtype=torch.bfloat16)
    ws = grass.step.GrassWorkspace([(m, n)], tokens, r, torch.bfloat16, grass.SEL_TOPR, device="cpu")
    ws.norms = ws.norms.as_subclass(OnGpu)
    kw = dict(dict(alpha=0.25, lr=1e-3), **kw)
    l = cls(W, r, grass.SEL_TOPR, K, workspace=ws, **kw)
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


KEPT, NOT_KEPT = dict(m=M, n=N, r=R, tokens=T), dict(m=4096, n=4096, r=R, tokens=256)


@pytest.mark.parametrize("shape", [KEPT, NOT_KEPT], ids=["kept", "not kept"])
@pytest.mark.parametrize("reset", [True, False])
def test_a_group_has_one_set_of_hyper_parameters_on_every_path(calls, shape, reset):
    """Layer 0's lr, betas, eps, alpha and step count go for the group, on a refresh of either kind as on
    a regular step; each layer keeps its own counters, epoch, layer id and reset flag."""
    assert B.grass_refresh_keeps_gradient(shape["tokens"], shape["m"], shape["n"], R, B.BF16) == (shape is KEPT)
    layers = [layer(**shape, lr=1e-3 * (g + 1), alpha=0.25 * (g + 1), beta1=0.9 - g / 10, eps=1e-8 * (g + 1),
                    layer_id=7 + g, reset_state=reset if g == 0 else not reset) for g in range(2)]
    for g, l in enumerate(layers):
        l.t, l.adam_step = 4 + 2 * g, 10 + g
    group = grass.step.GrassLayerGroup(layers, shape["tokens"], device="cpu")
    dYs, Xs = bf16(2, shape["tokens"], shape["m"]), bf16(2, shape["tokens"], shape["n"])
    group.step(dYs, Xs)
    first = 1 if reset else 11
    assert [l.adam_step for l in layers] == [first, 12 if reset else 1] and [l.t for l in layers] == [5, 7]
    if shape is KEPT:
        assert [c[0] for c in calls] == ["refresh", "refresh"]
        assert [(c[2]["layer_id"], c[2]["epoch"], bool(c[2]["reset_state"])) for c in calls] == \
            [(7, 2, reset), (8, 3, not reset)]
        assert [c[1]["W"][0] for c in calls] == [l.W.data_ptr() for l in layers]
        got = [(c[1]["lr"], c[1]["beta1"], c[1]["eps"], c[1]["alpha"], c[1]["step"]) for c in calls]
    else:
        assert [c[0] for c in calls[:4]] == ["grass_grad_row_norms", "grass_select"] * 2
        assert [c[1][5:7] for c in calls[1:4:2]] == [(7, 2), (8, 3)]
        # then the projection call, whose token slices a refresh keeps, and the update
        assert [c[0] for c in calls[4:]] == ["grass_project_grad_batched", "grass_adam_scatter_batched"]
        assert list(calls[4][1][11]) == [l.Gc.data_ptr() for l in layers]
        assert list(calls[5][1][7]) == [l.W.data_ptr() for l in layers]
        lr, beta1, _, eps, step, alpha = calls[5][1][15:21]
        got = [(lr, beta1, eps, alpha, step)]
    assert set(got) == {(1e-3, 0.9, 1e-8, 0.25, first)}
    group.step(dYs, Xs)
    assert calls[-1][0] == "step" and calls[-1][1]["count"] == 2
    assert (calls[-1][1]["lr"], calls[-1][1]["alpha"], calls[-1][1]["step"]) == (1e-3, 0.25, first + 1)


class OwnRows(grass.GrassLayer):
    """A program's own choice of rows."""

    def refresh(self, dY, X):
        self.refreshed = (dY, X)


@pytest.mark.parametrize("side", ["rows", "cols"])
def test_a_refresh_of_the_programs_own_is_called(calls, side):
    l = layer(cls=OwnRows) if side == "rows" else layer(m=N, n=N, cls=OwnRows, side="cols")
    dY, X = bf16(1, T, M if side == "rows" else N)[0], bf16(1, T, N)[0]
    l.step(dY, X)
    assert l.refreshed[0] is (dY if side == "rows" else X)
    assert [c[0] for c in calls] == ["grass_project_grad", "grass_subspace_adam",
                                     "grass_scatter_update" if side == "rows" else "grass_scatter_update_cols"]
    l.step(dY, X)
    assert calls[-1][0] == "step" and (l.t, l.adam_step) == (2, 2)


def test_a_groups_refresh_calls_the_layers_own(calls):
    layers = [layer(cls=OwnRows), layer(cls=OwnRows)]
    group = grass.step.GrassLayerGroup(layers, T, device="cpu")
    dYs, Xs = bf16(2, T, M), bf16(2, T, N)
    group.step(dYs, Xs)
    assert [l.refreshed[0] is dY for l, dY in zip(layers, dYs)] == [True, True]
    assert [c[0] for c in calls] == ["grass_project_grad_batched", "grass_adam_scatter_batched"]


def test_a_single_token_has_no_pitch(calls):
    """Views of one row differ in a stride that nothing uses; with more rows the layers must agree."""
    group = grass.step.GrassLayerGroup([layer(t=1), layer(t=1)], T, device="cpu")
    wide = gpu(4, M + 16, dtype=torch.bfloat16)
    group.step([wide[:1, :M], bf16(1, 1, M)[0]], [bf16(1, 1, N)[0], gpu(4, N + 8, dtype=torch.bfloat16)[1:2, :N]])
    assert calls[-1][1]["lddy"] == M + 16 and calls[-1][1]["T"] == 1
    for bad in ([wide[:2, :M], bf16(1, 2, M)[0]], [wide[:1, :M], bf16(1, 1, M + 1)[0]],
                [wide[:1, :M], gpu(M, 2, dtype=torch.bfloat16).T[:1]]):
        with pytest.raises(ValueError):
            group.step(bad, bf16(2, bad[0].shape[0], N))


def test_a_groups_buffers_are_looked_at_again_after_they_were_refused(calls):
    group = grass.step.GrassLayerGroup([layer(t=1, K=1 << 30), layer(t=1, K=1 << 30)], T, device="cpu")
    l, dYs, Xs = group.layers[1], bf16(2, T, M), bf16(2, T, N)
    V = l.V
    l.V = gpu(R, N, dtype=torch.float64)
    for _ in range(2):
        with pytest.raises(TypeError):
            group.step(dYs, Xs)
    l.V = V
    l.keep_U = False
    group.step(dYs, Xs)
    assert calls[-1][1]["V"][1] == V.data_ptr() and calls[-1][1]["U"][1] is None
    l.W.data = torch.zeros_like(l.W)                 # the same tensor, other memory
    group.step(dYs, Xs)
    assert calls[-1][1]["W"][1] == l.W.data_ptr()


@pytest.mark.parametrize("grouped", [False, True])
def test_a_refused_refresh_leaves_the_counters(calls, monkeypatch, grouped):
    layers = [layer() for _ in range(2 if grouped else 1)]
    for l in layers:
        l.t, l.adam_step = 4, 9
    stepper = grass.step.GrassLayerGroup(layers, T, device="cpu") if grouped else layers[0]
    args = (bf16(2, T, M), bf16(2, T, N)) if grouped else (bf16(1, T, M)[0], bf16(1, T, N)[0])
    library, entry = type(B.load_library()), "grass_refresh_step"
    good = library.__dict__[entry]
    monkeypatch.setattr(library, entry, staticmethod(lambda step, refresh, stream: 5))
    with pytest.raises(grass.GrassError):
        for l in layers:
            l._call = None
        stepper.step(*args)
    assert [(l.t, l.adam_step) for l in layers] == [(4, 9)] * len(layers)
    monkeypatch.setattr(library, entry, good)
    for l in layers:
        l._call = None
    stepper.step(*args)
    assert [(l.t, l.adam_step) for l in layers] == [(5, 1)] * len(layers) and calls[-1][1]["step"] == 1


@pytest.mark.parametrize("dY,X", [
    (gpu(T, M, M, dtype=torch.bfloat16), gpu(T, N, dtype=torch.bfloat16)),
    (gpu(T, M, dtype=torch.bfloat16), gpu(T, N, N, dtype=torch.bfloat16)),
    (gpu(M, T, dtype=torch.bfloat16).T, gpu(T, N, dtype=torch.bfloat16)),
    (gpu(T, 2 * M, dtype=torch.bfloat16)[:, ::2], gpu(T, N, dtype=torch.bfloat16)),
    (gpu(T, M, dtype=torch.bfloat16), gpu(T, N)), (gpu(T, M, dtype=torch.float16), gpu(T, N, dtype=torch.float16)),
    (gpu(T, M, dtype=torch.bfloat16), gpu(T + 1, N, dtype=torch.bfloat16)), (gpu(T, M - 1, dtype=torch.bfloat16),) * 2,
    (torch.zeros(T, M, dtype=torch.bfloat16), gpu(T, N, dtype=torch.bfloat16)),
], ids=str)
def test_inputs_of_another_form_are_refused(calls, dY, X):
    call = B.LayerStepCall()
    call.state(0, **buffers())
    with pytest.raises((ValueError, TypeError)):
        call.inputs(0, dY, X)


def test_pitches_reach_the_call(calls):
    wide = buffers()
    for name, pad in (("M", 3), ("V", 3), ("U", 3), ("Gc", 5)):
        wide[name] = gpu(R, N + pad)[:, :N]
    wide["W"] = gpu(M, N + 8, dtype=torch.bfloat16)[:, :N]
    call = B.LayerStepCall()
    call.state(0, **wide)
    call.inputs(0, gpu(T, M + 16, dtype=torch.bfloat16)[:, :M], gpu(T, N + 24, dtype=torch.bfloat16)[:, :N])
    a = call.args
    assert (a.ldstate, a.ldgc, a.ldw, a.lddy, a.ldx) == (N + 3, N + 5, N + 8, M + 16, N + 24)
    for name in ("M", "W", "Gc"):
        with pytest.raises(ValueError):
            B.LayerStepCall().state(0, **dict(buffers(), **{name: gpu(*wide[name].shape[::-1], dtype=wide[name].dtype).T}))


def test_the_scan_takes_only_tensors_alike_to_those_let_through():
    """accepted(): addresses are written only where shape, strides, dtype, device and which are None all agree; what is no
    plain tensor is left to the checks."""
    accepted = B._accepted()
    at = (ctypes.c_uint64 * (8 * 3))()
    where = ctypes.addressof(at)
    x, y = torch.zeros(4, 6), torch.zeros(8, dtype=torch.int32)
    seen = accepted(where, None, x, None, y)
    assert isinstance(seen, bytes) and not any(at)
    other = torch.ones(4, 6), None, torch.ones(8, dtype=torch.int32)
    assert accepted(where, seen, *other) is True
    assert (at[0], at[8], at[16]) == (other[0].data_ptr(), 0, other[2].data_ptr())
    was = list(at)
    for bad in ((x.T.contiguous().T, None, y), (torch.zeros(4, 7)[:, :6], None, y), (x.double(), None, y),
                (x, y, None), (x, x, y), (x, None, y[:7]), (x, None, torch.zeros(16, dtype=torch.int32)[::2]),
                (x.to("meta"), None, y)):
        assert accepted(where, seen, *bad) is not True and list(at) == was
    for odd in (gpu(4, 6), 3, torch.zeros(2, 2, 2), torch.zeros(4, 6).to_sparse()):
        assert accepted(where, seen, odd, None, y) is None and list(at) == was


def test_a_scanned_call_is_checked_again_when_layer_0_changes(calls, monkeypatch):
    """Other layers and the inputs go with layer 0's sizes: what was let through with one layer 0 is not with another."""
    plain = {k: torch.zeros(v.shape, dtype=v.dtype) for k, v in buffers().items()}
    monkeypatch.setattr(torch.Tensor, "is_cuda", True)
    call = B.LayerStepCall()
    for g in range(2):
        call.state(g, **plain)
        call.inputs(g, torch.zeros(T, M, dtype=torch.bfloat16), torch.zeros(T, N, dtype=torch.bfloat16))
    again = {k: v.clone() for k, v in plain.items()}
    call.state(1, **again)
    assert call.args.M[1] == again["M"].data_ptr() and call.args.W[0] == plain["W"].data_ptr()
    call.state(0, **{k: torch.zeros(v.shape, dtype=v.dtype) for k, v in buffers(r=R - 1).items()})
    assert call.args.r == R - 1
    with pytest.raises(ValueError):
        call.state(1, **again)
    call.state(0, **{k: torch.zeros(v.shape, dtype=v.dtype) for k, v in buffers(n=N + 8).items()})
    with pytest.raises(ValueError):
        call.inputs(0, torch.zeros(T, M, dtype=torch.bfloat16), torch.zeros(T, N, dtype=torch.bfloat16))
    with pytest.raises(ValueError):
        call.state(0, **plain, cols=True)


@pytest.fixture
def plain(calls, monkeypatch):
    """Tensors that the scan takes (it leaves subclasses to the checks) and that pass for CUDA tensors."""
    monkeypatch.setattr(torch.Tensor, "is_cuda", True)

    def plain_group(count=2, tokens=16):
        layers = [layer(t=1, K=1 << 30, tokens=tokens) for _ in range(count)]
        for l in layers:
            for name in ("W", "idx", "rho", "Gc", "M", "V", "U"):
                setattr(l, name, getattr(l, name).as_subclass(torch.Tensor))
        return grass.step.GrassLayerGroup(layers, tokens, device="cpu")

    return plain_group


def zeros(*shapes):
    return [torch.zeros(shape, dtype=torch.bfloat16) for shape in shapes]


@pytest.mark.parametrize("bad", [((4, M), (16, N)), ((16, M), (15, N)), ((16, M - 1), (16, N))],
                         ids=["few of dY", "few of X", "narrow"])
def test_inputs_go_with_the_ones_that_layer_0_was_let_through_with(calls, plain, bad):
    """Not with those that it was refused with: what goes with them would be read past its end."""
    group, good = plain(), zeros((16, M), (16, N))
    group.step([good[0]] * 2, [good[1]] * 2)
    refused = zeros(*bad)
    for g in range(2):                                   # as layer 0's, then as layer 1's
        pairs = [refused, good] if g == 0 else [good, refused]
        with pytest.raises(ValueError):
            group.step(*map(list, zip(*pairs)))
    assert len(calls) == 1
    group.step([good[0], gpu(16, M, dtype=torch.bfloat16)], [good[1], gpu(16, N, dtype=torch.bfloat16)])
    assert calls[-1][1]["T"] == 16 and len(calls) == 2


def test_a_single_token_of_another_pitch_goes_with_layer_0_after_a_refusal(calls, plain):
    group = plain()
    wide = zeros((4, M + 16))[0][:1, :M]
    group.step([zeros((1, M))[0], wide], zeros((1, N), (1, N)))
    with pytest.raises(ValueError):
        group.step(zeros((2, M), (1, M)), zeros((3, N), (1, N)))
    group.step([zeros((1, M))[0], wide], zeros((1, N), (1, N)))
    assert calls[-1][1]["dY"][1] == wide.data_ptr() and calls[-1][1]["T"] == 1


def test_a_layer_0_that_has_no_address_leaves_nothing_of_itself(calls, plain):
    """Its sizes are in the call by then: the layer 0 before it is checked, and put in, again."""
    class Nowhere(OnGpu):
        def data_ptr(self):
            raise RuntimeError("no storage")

    good = {k: torch.zeros(v.shape, dtype=v.dtype) for k, v in buffers().items()}
    call = B.LayerStepCall()
    call.state(0, **good)
    with pytest.raises(RuntimeError):
        call.state(0, **dict(buffers(r=R - 1), M=torch.zeros(R - 1, N).as_subclass(Nowhere)))
    call.state(0, **good)
    assert call.args.r == R and call.args.M[0] == good["M"].data_ptr()


@pytest.mark.parametrize("name,view", [("W", lambda t: t.view(torch.float16)), ("V", lambda t: t[:R - 1]),
                                       ("M", lambda t: t.view(R // 2, 2 * N)), ("idx", lambda t: t[:R - 1]),
                                       ("Gc", lambda t: t.view(torch.int32))], ids=["W", "V", "M", "idx", "Gc"])
def test_a_groups_buffer_of_another_form_at_the_same_address_is_refused(calls, plain, name, view):
    group = plain()
    inputs = zeros((16, M), (16, M)), zeros((16, N), (16, N))
    group.step(*inputs)
    held, l = getattr(group.layers[1], name), group.layers[1]
    setattr(l, name, view(held))
    assert getattr(l, name).data_ptr() == held.data_ptr()
    with pytest.raises((TypeError, ValueError)):
        group.step(*inputs)
    setattr(l, name, held)
    group.step(*inputs)
    assert len(calls) == 2
