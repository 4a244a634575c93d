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
