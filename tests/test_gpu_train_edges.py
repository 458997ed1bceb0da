"""Gradients at the edges of the backward kernels' tiles: batches of one 8-row group, one group past
a block of rows, and several blocks with a remainder; layer widths below, at and past the column
blocks.  Every entry against the oracle's BF16-storage-emulated backward.

Bound: 2^-7 of the sum of the terms' magnitudes (gradcheck.py), with the layer's mean |delta| added
to every |delta|: in a batch of 8 rows a delta that is itself a cancelling sum moves by more than a
BF16 unit of its own value when one of its terms rounds the other way, but not by more than a BF16
unit of its terms.  An 8-row group lost or counted twice at an edge is at least 1/97 of the sum.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import gradcheck  # noqa: E402
from oracle import mlp  # noqa: E402
from paper_2402_18858_gb300 import workload as w  # noqa: E402


@pytest.mark.parametrize("hidden,B", [([16, 8], 8), ([24, 40], 136), ([136, 72], 264), ([264, 24], 520),
                                      ([1600, 48], 648), ([48, 272], 776)])
def test_gradients_at_tile_edges(mechs, hidden, B):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2402_18858_gb300 import build, chem as lc
    build.build()
    m, path = mechs["c_30"]
    gm = lc.chem_load_mech(path)
    ann = lc.chem_ann_create(gm, hidden, seed=11)
    st = w.make_states(m, B, 77)
    T, p, Y0 = (torch.as_tensor(a, device="cuda") for a in (st.T, st.p, st.Y))
    noise = torch.as_tensor(np.random.default_rng(2).standard_normal(st.Y.shape), device="cuda")
    Y1 = (Y0 * (1.0 + 0.01 * noise)).contiguous()
    lc.chem_ann_fit_norm(ann, T, p, Y0, Y1)
    X = torch.empty((B, 64), dtype=torch.bfloat16, device="cuda")
    bcty = torch.empty((B, m.n_species), dtype=torch.float32, device="cuda")
    lc.chem_ann_features(ann, T, p, Y0, X, bcty=bcty)
    U = torch.empty((B, ann.n_out_pad), dtype=torch.float32, device="cuda")
    lc.chem_ann_targets(ann, Y0, Y1, U)
    lc.chem_ann_train_step(ann, X, U, bcty, apply=False)
    torch.cuda.synchronize()
    assert lc.chem_ann_error(ann) == 0
    grads = mlp.unflatten(lc.chem_ann_get_params(ann, which=1), ann.dims)
    params = mlp.unflatten(lc.chem_ann_get_params(ann), ann.dims)
    norm = lc.chem_ann_get_norm(ann).astype(np.float64)
    K, n_in = m.n_species, ann.n_in
    om, osd = norm[4 * n_in:4 * n_in + K], norm[4 * n_in + K:4 * n_in + 2 * K]
    x = X.float().cpu().numpy().astype(np.float64)
    Up, cache = mlp.forward(params, x, bf16=True)
    _, _, _, dU = mlp.loss_and_grad(Up, U.cpu().numpy().astype(np.float64), K, bcty.cpu().numpy().astype(np.float64),
                                    om, osd, 1.0, 0.1)
    ref, deltas = mlp.backward(params, cache, dU, bf16=True, with_deltas=True)
    for l, ((gw, gb), (ow, ob)) in enumerate(zip(grads, ref)):
        d = np.abs(deltas[l]) + np.abs(deltas[l]).mean()
        assert (np.abs(gw - ow) <= gradcheck.C * (d.T @ np.abs(cache[0][l])) + 1e-30).all(), l
        assert (np.abs(gb - ob) <= gradcheck.C * d.sum(axis=0) + 1e-30).all(), l
