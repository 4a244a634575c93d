"""Layers and groups of layers stepped as a training program does, against the separate library calls
and the fp64 oracle."""
import numpy as np
import pytest
import torch

import paper_2406_17660_b200 as grass
from paper_2406_17660_b200 import synthetic as syn

pytestmark = pytest.mark.gpu
DEV = "cuda"
BF16 = torch.bfloat16


def rel(a, b):
    a, b = a.double(), b.double()
    return float((a - b).norm() / b.norm())


def inputs(T, m, n, seed=0, proj=0, dtype=BF16):
    """dY, X and W of one layer on the device, each with a pitch that is a multiple of eight elements."""
    dY, X = (syn._padded(f(T, k, dtype, seed0=seed, proj=proj).to(DEV), syn.pad_to(k, 8))
             for f, k in ((syn.make_dY, m), (syn.make_X, n)))
    return dY, X, syn._padded(syn.make_W(m, n, dtype, seed0=seed, proj=proj).to(DEV), syn.pad_to(n, 8))


def rows_of(m, r, seed=0):
    return torch.tensor(np.sort(np.random.default_rng(seed).choice(m, r, replace=False)), dtype=torch.int32,
                        device=DEV)


@pytest.mark.parametrize("count,Tmax,T,m,n,r", [
    (1, 16384, 16128, 512, 512, 64), (1, 4096, 3840, 1024, 1024, 256), (1, 4096, 4003, 2048, 2048, 128),
    (4, 4096, 3840, 512, 512, 64), (4, 4096, 3072, 300, 328, 128),
])
def test_a_short_batch_runs_in_the_workspace_of_a_longer_one(count, Tmax, T, m, n, r):
    """The last, shorter batch of an epoch: its own tiling may want more slices than the workspace holds."""
    layers, dYs, Xs = [], [], []
    ws = grass.step.GrassWorkspace([(m, n)], Tmax, r, BF16, grass.SEL_TOPR)
    for g in range(count):
        dY, X, W = inputs(T, m, n, proj=g)
        l = grass.GrassLayer(W, r, grass.SEL_TOPR, 1 << 30, 0.25, 1e-3, workspace=ws)
        l.idx.copy_(rows_of(m, r, g)); l.t = 1
        layers.append(l); dYs.append(dY); Xs.append(X)
    if count == 1:
        layers[0].step(dYs[0], Xs[0])
    else:
        grass.step.GrassLayerGroup(layers, Tmax).step(dYs, Xs)
    grass.grass_device_status()
    full = torch.empty(grass.grass_project_workspace_bytes(T, m, n, r, grass.BF16), dtype=torch.uint8, device=DEV)
    for l, dY, X in zip(layers, dYs, Xs):
        want = torch.empty_like(l.Gc)
        grass.grass_project_grad(dY, X, l.idx, l.rho, r, want, full)
        assert rel(l.Gc, want) <= 1e-5


def test_a_step_over_millions_of_tokens():
    """More tokens than the separate gather takes (2 097 120): the cooperative one does them."""
    T, m, n, r = 2_200_000, 1024, 512, 256
    g = torch.Generator(device=DEV).manual_seed(1)
    dY, X = (torch.empty((T, k), dtype=BF16, device=DEV).normal_(generator=g) for k in (m, n))
    ws = grass.step.GrassWorkspace([(m, n)], T, r, BF16, grass.SEL_TOPR)
    l = grass.GrassLayer(torch.zeros((m, n), dtype=BF16, device=DEV), r, grass.SEL_TOPR, 1 << 30, 0.25, 1e-3,
                         workspace=ws)
    l.idx.copy_(rows_of(m, r)); l.t = 1
    l.step(dY, X)
    grass.grass_device_status()
    want = torch.zeros((r, n), dtype=torch.float64, device=DEV)
    for t in range(0, T, 100_000):
        want += dY[t:t + 100_000, l.idx.long()].double().T @ X[t:t + 100_000].double()
    assert rel(l.Gc, want) <= 1e-4


@pytest.mark.parametrize("dtype", [BF16, torch.float32], ids=["bf16", "fp32"])
@pytest.mark.parametrize("lengths", [(1, 2, 30, 7), (31, 2, 100, 1, 63), (33,), (200,), (5,) * 20])
def test_the_column_form_rounds_as_the_column_scatter(dtype, lengths):
    """Columns drawn several times, their runs crossing blocks of 32: the one-call update leaves the same bits
    as Adam and the column scatter of the same G_C."""
    T, m, n, r = 256, 300, 77, sum(lengths)
    rng = np.random.default_rng(r)
    X, dY = (syn._padded(f(T, k, dtype, seed0=6).to(DEV), syn.pad_to(k, 8))
             for f, k in ((syn.make_X, m), (syn.make_dY, n)))
    W0 = syn._padded(syn.make_W(n, m, dtype, seed0=6).to(DEV), syn.pad_to(m, 8))
    cols = np.repeat(np.sort(rng.choice(m, len(lengths), replace=False)), lengths)
    ws = grass.step.GrassWorkspace([(m, n)], T, r, dtype, grass.SEL_TOPR)
    l = grass.GrassLayer(W0.clone(), r, grass.SEL_TOPR, 1 << 30, 0.25, 1e-3, workspace=ws, side="cols")
    l.idx.copy_(torch.tensor(cols, dtype=torch.int32)); l.t, l.adam_step = 1, 3
    l.rho.copy_(torch.tensor(0.5 + rng.random(r), dtype=torch.float32))
    l.M.normal_(); l.V.uniform_(0.5, 1.5)
    M, V, U, W = l.M.clone(), l.V.clone(), torch.empty_like(l.U), W0.clone()
    l.step(dY, X)
    grass.grass_subspace_adam(l.Gc, M, V, U, l.lr, l.beta1, l.beta2, l.eps, 4)
    grass.grass_scatter_update_cols(W, U, l.idx, l.rho, l.alpha)
    grass.grass_device_status()
    for name, want in (("M", M), ("V", V), ("U", U), ("W", W)):
        assert torch.equal(getattr(l, name), want), name


@pytest.mark.parametrize("m,n", [(37, 4), (300, 91), (65, 128), (129, 129), (700, 203), (50, 256), (33, 257), (90, 512),
                                 (21, 513), (40, 1030)])
@pytest.mark.parametrize("dtype", [BF16, torch.float32], ids=["bf16", "fp32"])
def test_norms_of_short_rows(m, n, dtype):
    """Row norms from split partials, at the row lengths where the number of rows a CTA takes changes; the rows
    past the last do not reach the norms."""
    T = 4096
    dY, X, _ = inputs(T, m, n, seed=5, dtype=dtype)
    code = grass.BF16 if dtype == BF16 else grass.F32
    ws = torch.full((grass.grass_grad_row_norms_workspace_bytes(T, m, n, code),), 0x7F, dtype=torch.uint8, device=DEV)
    norms = torch.full((m + 64,), -1.0, device=DEV)
    grass.grass_grad_row_norms(dY, X, norms[:m], ws)
    grass.grass_device_status()
    want = (dY.double().T @ X.double()).norm(dim=1)
    # exact products, fp32 sums over 4096 tokens in slices and n columns
    assert float(((norms[:m].double() - want).abs() / want).max()) <= 1e-5
    assert bool((norms[m:] == -1).all())


@pytest.mark.parametrize("r,n", [(585, 1024), (586, 1024), (146, 4096), (147, 4096), (109, 5461), (110, 5461)])
@pytest.mark.parametrize("repeats", [False, True])
def test_update_forms_around_their_limits(r, n, repeats):
    """Elements just below and above where the update changes its kernel: the bits of Adam and the row scatter."""
    rng = np.random.default_rng(r + n)
    m = 2 * r
    idx = torch.tensor(np.sort(rng.choice(m, r, replace=False) if not repeats else (rng.pareto(1.0, r) * 8).astype(int) % m),
                       dtype=torch.int32, device=DEV)
    rho, Gc = torch.rand(r, device=DEV) + 0.5, torch.randn((r, n), device=DEV)
    M, V, W = torch.randn((r, n), device=DEV), torch.rand((r, n), device=DEV), torch.randn((m, n), device=DEV).to(BF16)
    want = [t.clone() for t in (M, V, W)]
    U, hp = torch.empty_like(M), (1e-3, 0.9, 0.999, 1e-8, 3)
    grass.grass_subspace_adam(Gc, want[0], want[1], U, *hp)
    grass.grass_scatter_update(want[2], U, idx, rho, 0.25)
    grass.grass_adam_scatter(Gc, M, V, None, W, idx, rho, *hp, 0.25)
    grass.grass_device_status()
    for got, w in zip((M, V, W), want):
        assert torch.equal(got, w)


def layers_of(count, T, m, n, r, K=1 << 30, t=1, reset=True, seed=0):
    """`count` layers of one shape in mid-epoch, and their inputs."""
    ws = grass.step.GrassWorkspace([(m, n)], T, r, BF16, grass.SEL_TOPR)
    layers, dYs, Xs = [], [], []
    for g in range(count):
        dY, X, W = inputs(T, m, n, seed=seed, proj=g)
        l = grass.GrassLayer(W, r, grass.SEL_TOPR, K, 0.25, 1e-3, reset_state=reset, seed=3, layer_id=g, workspace=ws)
        l.idx.copy_(rows_of(m, r, g))
        l.rho.copy_(torch.rand(r, generator=torch.Generator().manual_seed(g)) + 0.5)
        l.M.normal_(); l.V.uniform_(0.5, 1.5)
        l.t, l.adam_step = t, 6
        layers.append(l); dYs.append(dY); Xs.append(X)
    return layers, dYs, Xs


def state_of(layers):
    return [[getattr(l, k).clone() for k in ("M", "V", "U", "W")] for l in layers]


def check_update(layers, before, step):
    """M, V, U and W are those of the separate update from the layers' own G_C, bit for bit."""
    for l, (M, V, U, W) in zip(layers, before):
        grass.grass_adam_scatter(l.Gc, M, V, U, W, l.idx, l.rho, l.lr, l.beta1, l.beta2, l.eps, step, l.alpha)
        for k, want in (("M", M), ("V", V), ("U", U), ("W", W)):
            assert torch.equal(getattr(l, k), want), k


MODES = [
    # layers, T, m, n, r, and what the step's own plan picks: gather, pair, short slices
    (1, 1000, 256, 256, 100, grass.GATHER_PREPASS, 0, False),
    (1, 3000, 1024, 2048, 1024, grass.GATHER_PREPASS, 1, False),
    (2, 9000, 1024, 5461, 1024, grass.GATHER_PREPASS, 1, True),
    (1, 1000, 256, 256, 64, grass.GATHER_IN_CTA, 0, True),
    (4, 3000, 256, 256, 256, grass.GATHER_IN_CTA, 1, True),
    (1, 6000, 4096, 5461, 1024, grass.GATHER_COOPERATIVE, 1, False),
    (1, 9000, 4096, 5461, 512, grass.GATHER_COOPERATIVE, 1, False),
]


@pytest.mark.parametrize("count,T,m,n,r,gather,pair,short", MODES)
def test_every_gather_hands_over_to_the_update(count, T, m, n, r, gather, pair, short):
    """Each gather, single CTAs and pairs, long and short slices, followed by the update in one call, eagerly and
    from a CUDA graph: G_C of the projection calls to summation order, the update's bits."""
    p = grass.grass_step_plan(count, T, m, n, r)
    assert (p["gather"], p["cta_pair"], p["short_slices"] > 0) == (gather, pair, short)
    layers, dYs, Xs = layers_of(count, T, m, n, r)
    stepper = layers[0] if count == 1 else grass.step.GrassLayerGroup(layers, T)
    args = (dYs[0], Xs[0]) if count == 1 else (dYs, Xs)
    before = state_of(layers)
    stepper.step(*args)
    grass.grass_device_status()
    full = torch.empty(grass.grass_project_batched_workspace_bytes(count, T, m, n, r), dtype=torch.uint8, device=DEV)
    want = [torch.empty_like(l.Gc) for l in layers]
    grass.grass_project_grad_batched(dYs, Xs, [l.idx for l in layers], [l.rho for l in layers], r, want, full)
    for l, w in zip(layers, want):
        assert rel(l.Gc, w) <= 1e-5
    check_update(layers, before, 7)
    eager = [l.Gc.clone() for l in layers]
    before = state_of(layers)
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        stepper.step(*args)
    graph.replay()
    grass.grass_device_status()
    for l, g in zip(layers, eager):
        assert torch.equal(l.Gc, g)
    check_update(layers, before, 8)


@pytest.mark.parametrize("reset", [True, False])
@pytest.mark.parametrize("T,m,n,r,kept", [(4096, 512, 520, 100, True), (256, 4096, 4100, 200, False)])
def test_a_group_against_its_layers_stepped_singly(T, m, n, r, kept, reset):
    """A refresh that keeps its gradient has the bits of the layers' own; one that does not, those of the batched
    projection; then a regular step."""
    assert grass.grass_refresh_keeps_gradient(T, m, n, r, grass.BF16) == kept
    (grouped, dYs, Xs), (single, _, _) = (layers_of(3, T, m, n, r, K=4, t=4, reset=reset) for _ in range(2))
    for a, b in zip(grouped, single):
        b.M.copy_(a.M); b.V.copy_(a.V)
    before = state_of(grouped)
    group = grass.step.GrassLayerGroup(grouped, T)
    group.step(dYs, Xs)
    for l, dY, X in zip(single, dYs, Xs):
        l.step(dY, X)
    grass.grass_device_status()
    for a, b in zip(grouped, single):
        assert torch.equal(a.idx, b.idx) and torch.equal(a.rho, b.rho)
        assert (a.t, a.adam_step) == (b.t, b.adam_step) == (5, 1 if reset else 7)
        assert rel(a.Gc, b.Gc) <= 1e-5
        if kept:
            for k in ("Gc", "M", "V", "U", "W"):
                assert torch.equal(getattr(a, k), getattr(b, k)), k
    if not kept:
        want = [torch.empty_like(l.Gc) for l in grouped]
        grass.grass_project_grad_batched(dYs, Xs, [l.idx for l in grouped], [l.rho for l in grouped], r, want, group.ws)
        for l, w in zip(grouped, want):
            assert torch.equal(l.Gc, w)
    if reset:
        for b in before:
            b[0].zero_(); b[1].zero_()
    check_update(grouped, before, 1 if reset else 7)
    before = state_of(grouped)
    group.step(dYs, Xs)
    check_update(grouped, before, 2 if reset else 8)


@pytest.mark.parametrize("count,T,m,n,r", [
    (4, 32768, 4096, 4096, 1024), (2, 32768, 11008, 4096, 256),     # 7B q,k,v,o and gate,up
    (1, 65536, 2048, 5461, 512), (2, 65536, 5461, 2048, 64),        # 1B down and gate,up
    (1, 65536, 1024, 2736, 256), (4, 65536, 512, 512, 128),         # 350M down, 60M q,k,v,o
    (1, 4096, 5120, 13824, 1024),                                   # 13B down, one micro-batch
])
def test_regular_steps_at_full_size(count, T, m, n, r):
    """The tiling that regular steps run at the LLaMA shapes, on sampled rows in 64 bits, and its update."""
    ws = grass.step.GrassWorkspace([(m, n)], T, r, BF16, grass.SEL_TOPR)
    layers, dYs, Xs = [], [], []
    gen = torch.Generator(device=DEV).manual_seed(T + m)
    for g in range(count):
        dY, X = (torch.empty((T, syn.pad_to(k, 8)), dtype=BF16, device=DEV).normal_(generator=gen)[:, :k] for k in (m, n))
        W = torch.empty((m, syn.pad_to(n, 8)), dtype=BF16, device=DEV).normal_(generator=gen)[:, :n]
        l = grass.GrassLayer(W, r, grass.SEL_TOPR, 1 << 30, 0.25, 1e-3, layer_id=g, workspace=ws)
        l.idx.copy_(rows_of(m, r, g)); l.t = 1
        l.V.fill_(1.0)
        layers.append(l); dYs.append(dY); Xs.append(X)
    before = state_of(layers)
    if count == 1:
        layers[0].step(dYs[0], Xs[0])
    else:
        grass.step.GrassLayerGroup(layers, T).step(dYs, Xs)
    grass.grass_device_status()
    for l, dY, X in zip(layers, dYs, Xs):
        js = torch.randint(r, (4,), device=DEV, generator=gen)
        want = sum(dY[t:t + 8192][:, l.idx[js].long()].double().T @ X[t:t + 8192].double() for t in range(0, T, 8192))
        assert rel(l.Gc[js], want) <= 1e-4
        assert float((l.Gc[js] - want).abs().max() / want.abs().max()) <= 1e-4
    check_update(layers, before, 1)


@pytest.mark.parametrize("T", [1, 31, 65, 200])
@pytest.mark.parametrize("r", [1, 64, 65, 128, 129, 192, 257, 320])
@pytest.mark.parametrize("m", [330, 3400], ids=["dense", "sparse"])
def test_the_separate_gather_copies_what_the_cooperative_one_does(T, r, m):
    """Widths and token counts at which the separate gather has lanes, column groups or tokens to spare: the operand,
    hence G_C, has the bits of the cooperative gather."""
    n = 136
    dY, X, _ = inputs(T, m, n)
    idx = rows_of(m, r)
    out = []
    for gather in (grass.binding.GATHER_PREPASS, grass.binding.GATHER_COOPERATIVE):
        opts = dict(gather=gather, token_slices=1, cta_pair=1, n_blocks_per_cta=1)
        ws = torch.empty(grass.grass_project_plan(1, T, m, n, r, opts)["workspace_bytes"], dtype=torch.uint8, device=DEV)
        ws.fill_(0x7f)
        Gc = torch.empty((r, n), device=DEV)
        grass.binding.grass_project_grad_ex([dY], [X], [idx], [None], r, [Gc], ws, opts)
        out.append(Gc)
    grass.grass_device_status()
    want = dY[:, idx.long()].double().T @ X.double()
    assert torch.equal(*out) and rel(out[0], want) <= 1e-5


@pytest.mark.parametrize("shape", [(2048, 512, 512, 128), (2048, 1024, 512, 256), (4096, 512, 256, 128)])
@pytest.mark.parametrize("gather", [grass.binding.GATHER_AUTO, grass.binding.GATHER_PREPASS,
                                    grass.binding.GATHER_COOPERATIVE, grass.binding.GATHER_IN_CTA])
def test_a_projection_waits_for_the_kernel_that_makes_its_inputs(shape, gather):
    """The first kernel of a call is placed while the program's kernel before it drains: what that one writes (here new
    dY and X on every iteration, right before the call) is what the projection reads, eagerly and in a graph
    that forks and joins streams before the call."""
    T, m, n, r = shape
    r = 64 if gather == grass.binding.GATHER_IN_CTA else r
    base_dY, base_X, _ = inputs(T, m, n)
    dY, X = torch.zeros_like(base_dY), torch.zeros_like(base_X)
    idx, opts = rows_of(m, r), dict(gather=gather)
    ws = torch.empty(grass.grass_project_plan(1, T, m, n, r, opts)["workspace_bytes"], dtype=torch.uint8, device=DEV)
    Gc, want = torch.empty((r, n), device=DEV), torch.empty((r, n), device=DEV)

    def project(a, b, out):
        grass.binding.grass_project_grad_ex([a], [b], [idx], [None], r, [out], ws, opts)

    project(base_dY, base_X, want)
    seen = []
    for k in range(30):                                    # powers of two: exact in bf16 and fp32
        torch.mul(base_dY, 2.0 ** (k % 5), out=dY)
        torch.mul(base_X, 2.0 ** -(k % 3), out=X)
        project(dY, X, Gc)
        seen.append((Gc.clone(), 2.0 ** (k % 5 - k % 3)))
    for got, scale in seen:
        assert torch.equal(got, want * scale)
    main, side = torch.cuda.Stream(), torch.cuda.Stream()
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=main):
        side.wait_stream(main)
        with torch.cuda.stream(side):
            dY.copy_(base_dY)
        X.zero_()
        X.add_(base_X)
        main.wait_stream(side)
        project(dY, X, Gc)
        dY.mul_(2.0)
        project(dY, X, Gc)
    for _ in range(3):
        Gc.zero_()
        dY.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(Gc, want * 2.0)
    grass.grass_device_status()


def test_row_norms_and_selection_wait_for_the_kernel_before():
    G, norms = torch.empty((3000, 700), device=DEV), torch.empty(3000, device=DEV)
    idx, rho = torch.zeros(64, dtype=torch.int32, device=DEV), torch.zeros(64, device=DEV)
    for k in range(20):
        G.fill_(0.0)
        G[k:k + 64] = 2.0 ** k
        grass.grass_row_norms(G, norms)
        grass.grass_select(norms, 64, grass.SEL_TOPR, 0, 0, 0, idx, rho, None)
        assert torch.equal(idx.long(), torch.arange(k, k + 64, device=DEV))
    grass.grass_device_status()


@pytest.mark.parametrize("T,m,n,r,side,gather", [
    (2048, 512, 512, 128, "rows", grass.GATHER_PREPASS), (4096, 512, 256, 64, "rows", grass.GATHER_IN_CTA),
    (1024, 1024, 2736, 256, "rows", grass.GATHER_PREPASS), (6000, 4096, 5461, 1024, "rows", grass.GATHER_COOPERATIVE),
    (2048, 1376, 512, 128, "cols", None), (512, 256, 256, 32, "rows", None),
], ids=["narrow", "narrow in-CTA", "wide", "wide cooperative", "cols", "fp32"])
def test_a_step_waits_for_the_kernels_that_write_its_state(T, m, n, r, side, gather):
    """A program may write rows, scales, state and weights right before a regular step (a checkpoint loaded, rows of its
    own): the update is that of what it wrote last, whichever of them that is, eagerly and in a graph."""
    dtype = torch.float32 if T == 512 else BF16
    if gather is not None:
        assert grass.grass_step_plan(1, T, m, n, r)["gather"] == gather
    dY, X, W = inputs(T, m, n, dtype=dtype)
    rows, contract = (n, m) if side == "cols" else (m, n)
    ws = grass.step.GrassWorkspace([(rows, contract)], T, r, dtype, grass.SEL_TOPR)
    l = grass.GrassLayer(W, r, grass.SEL_TOPR, 1 << 30, 0.25, 1e-3, workspace=ws, side=side)
    g = torch.Generator(device=DEV).manual_seed(r)
    names = ("idx", "rho", "M", "V", "W")

    def written(seed):
        rho, V = (torch.rand(s, device=DEV, generator=g) + 0.5 for s in (r, (r, contract)))
        return dict(idx=rows_of(rows, r, seed), rho=rho, V=V, M=torch.randn((r, contract), device=DEV, generator=g),
                    W=(W.float() * (seed + 1)).to(dtype))

    def step(put, last=0):
        for k in names[last:] + names[:last]:
            torch.mul(put[k], 1, out=getattr(l, k))          # (a kernel, where copy_ may be a copy)
        l.t, l.adam_step = 1, 3
        l.step(dY, X)

    states, want = [written(0), written(1)], []
    for put in states:
        for k in names:
            getattr(l, k).copy_(put[k])
        torch.cuda.synchronize()
        l.t, l.adam_step = 1, 3
        l.step(dY, X)
        torch.cuda.synchronize()
        want.append([getattr(l, k).clone() for k in ("Gc", "M", "V", "U", "W")])
    assert not torch.equal(want[0][4], want[1][4])
    seen = []
    for k in range(20):
        step(states[k % 2], k // 2 % len(names))
        seen.append([getattr(l, k).clone() for k in ("Gc", "M", "V", "U", "W")])
    for k, got in enumerate(seen):
        assert all(torch.equal(a, b) for a, b in zip(got, want[k % 2])), k
    graph, stream = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=stream):
        for k in range(2 * len(names) + 1):
            step(states[k % 2], k // 2 % len(names))
    for _ in range(3):
        graph.replay()
        torch.cuda.synchronize()
        assert all(torch.equal(getattr(l, k), b) for k, b in zip(("Gc", "M", "V", "U", "W"), want[0]))
    grass.grass_device_status()
