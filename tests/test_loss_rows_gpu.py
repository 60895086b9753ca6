"""The detection loss at the edges of its tiles (256 threads x 15 boxcar
starts): rows shorter than a tile, one start more or less than a whole one,
and several; a tie between two starts of one row and of two."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
TILE = 256 * 15


@pytest.mark.parametrize("n_cols", [8, 9, 14, 15, 22, TILE + 6, TILE + 7, TILE + 8, 2 * TILE + 7, 2 * TILE + 400])
def test_tile_edges_match_oracle(n_cols):
    from paper_1601_01165_gb300 import binding as dd
    rng = np.random.default_rng(n_cols)
    x = rng.standard_normal((5, n_cols)).astype(np.float32) + 3.0
    big = torch.full((5, n_cols + 3), 77.0, device="cuda")
    xt = big[:, :n_cols]
    xt.copy_(torch.from_numpy(x))
    raw, grad = dd.boxcar_snr(xt, grad=True)
    res = dd.snr_result(raw)
    if n_cols == 8:          # one boxcar a row: no deviation, no S/N (the oracle refuses)
        assert res["valid"] == 0 and not grad.cpu().numpy().any()
        return
    o = x.astype(np.float64)
    loss, g_ref, (bi, bt) = oracle.boxcar_snr_loss(o)
    assert res["valid"] == 1 and (res["best_row"], res["best_t"]) == (bi, bt)
    assert abs(res["loss"] - loss) <= 1e-9 * abs(loss)
    g = grad.cpu().numpy().astype(np.float64)
    assert g.shape == g_ref.shape and np.abs(g - g_ref).max() <= 1e-6 * np.abs(g_ref).max()


@pytest.mark.parametrize("gap", [3, 15, TILE])
def test_first_of_equal_starts(gap):
    """The same burst at two starts of a row, and the same row twice: the first counts."""
    from paper_1601_01165_gb300 import binding as dd
    x = torch.zeros((3, 3 * TILE), device="cuda")
    x[:, 1::2] = 0.5
    x[1:, 40:42] += 16.0
    x[1:, 40 + 2 * ((gap + 1) // 2) + 10:][:, :2] += 16.0
    res = dd.snr_result(dd.boxcar_snr(x)[0])
    b = x[1].double().unfold(0, 8, 1).sum(1)
    assert (res["best_row"], res["best_t"]) == (1, int((b == b.max()).nonzero()[0]))
