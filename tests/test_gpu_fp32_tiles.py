"""GPU parity of the tiled fp32 linear and attention kernels at the edges of
their tiles, K slices, key tiles and group split, with rows that are and are
not 16-byte aligned, against the CPU oracle."""

import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

DEV = "cuda"
EPS = 2.0 ** -24


@pytest.fixture(scope="module")
def acid():
    import __graft_entry__ as g

    g.build()
    from paper_2607_12358_gb300 import acid as a

    return a


def _t(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).to(DEV)


# key tiles of 32 in four groups: one key, groups without a tile, a ragged last
# tile, several tiles a group; query tiles of 16 rows (few heads) and 32
# rows (640 x 8: 160 tiles)
@pytest.mark.parametrize("nq,nk,H", [(1, 1, 1), (17, 31, 2), (33, 33, 3), (16, 64, 1), (47, 128, 2), (64, 129, 2),
                                     (100, 300, 4), (640, 65, 8)])
@pytest.mark.parametrize("D", [32, 64, 96, 128])
@pytest.mark.parametrize("pad", [0, 1])
def test_attention_fp32_tiles(acid, nq, nk, H, D, pad):
    rng = np.random.default_rng(nq + nk + D)
    w = H * D
    q, k, v = (rng.normal(size=(n, w + pad)).astype(np.float32) for n in (nq, nk, nk))
    q[:, pad:] *= 3.0  # scores of a few tens at head dim 128: the running max moves
    got = acid.acid_attention_forward(*(_t(x)[:, pad:] for x in (q, k, v)), H).cpu().numpy()
    qs, ks, vs = (x[:, pad:].reshape(len(x), H, D) for x in (q, k, v))
    ref = O.attention(qs, ks, vs).reshape(nq, w)
    # a score's rounding error, at most (D + 2) 2^-24 sum |q k| / sqrt(D), moves
    # its weight by that factor; weights and values then add nk + 8 roundings
    mag = np.abs(qs).astype(np.float64).max() * np.abs(ks).max() * np.sqrt(D)
    tol = (2 * (D + 2) * mag + nk + 8) * EPS * np.abs(vs).max()
    assert np.abs(got - ref).max() <= tol
    assert np.linalg.norm(got - ref) <= 1e-5 * np.linalg.norm(ref)


def test_attention_fp32_overflowing_scores(acid):
    """Keys whose scores are -inf get no weight, also when a whole key tile or
    a group's whole share is such keys."""
    D, nk = 64, 200
    rng = np.random.default_rng(5)
    q = np.full((20, D), 1e19, np.float32)
    k = np.full((nk, D), -1e20, np.float32)
    live = [40, 41, 150]
    k[live] = 0.0
    v = rng.normal(size=(nk, D)).astype(np.float32)
    got = acid.acid_attention_forward(_t(q), _t(k), _t(v), 1).cpu().numpy()
    assert np.allclose(got, v[live].mean(0), rtol=1e-5, atol=1e-6)
