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


# tiles of 16 x 32, 32 x 32 and 64 x 64 outputs by the number of tiles;
# K slices of 32 in four groups: one slice, fewer slices than groups, a ragged
# last slice, K not a multiple of 4 (4-byte copies)
@pytest.mark.parametrize("M,K,N", [(1, 32, 2), (15, 31, 34), (17, 8, 30), (16, 64, 32), (33, 127, 64), (256, 256, 768),
                                   (257, 100, 1026), (1000, 160, 770), (2049, 66, 514), (64, 4100, 96)])
@pytest.mark.parametrize("epi", ["bias", "gelu", "gated_res", "res"])
def test_linear_fp32_tiles(acid, M, K, N, epi):
    rng = np.random.default_rng(M + 3 * K + 7 * N)
    a, w = rng.normal(size=(M, K)).astype(np.float32), (0.1 * rng.normal(size=(N, K))).astype(np.float32)
    b, g = rng.normal(size=N).astype(np.float32), rng.normal(size=N).astype(np.float32)
    r = rng.normal(size=(M, N)).astype(np.float32)
    res = _t(r) if epi in ("gated_res", "res") else None
    got = acid.acid_linear_forward(_t(a), _t(w), _t(b), epilogue=epi, gate=_t(g), residual=res, out=res).cpu().numpy()
    acc = O.linear(a, w, b)
    ref = {"bias": acc, "gelu": O.gelu_tanh(acc), "gated_res": r + g * acc, "res": r + acc}[epi]
    # rounding of K products and additions: at most (K + 8) 2^-24 of the sum
    # of the terms' magnitudes (a few roundings more in the epilogue; GELU's
    # slope is below 1.13 and the gate scales the sum)
    mag = np.abs(a).astype(np.float64) @ np.abs(w).astype(np.float64).T + np.abs(b) + 1.0
    if epi == "gated_res":
        mag = mag * np.abs(g) + 1.0
    if epi in ("gated_res", "res"):
        mag = mag + np.abs(r)
    assert np.all(np.abs(got - ref) <= 1.13 * (K + 16) * EPS * mag)


def test_linear_fp32_strided_unaligned_rows(acid):
    """A with an odd row stride and out and residual rows at 4-byte offsets."""
    M, K, N = 70, 96, 66
    rng = np.random.default_rng(3)
    a, w = rng.normal(size=(M, K + 5)).astype(np.float32), rng.normal(size=(N, K)).astype(np.float32)
    buf = torch.zeros(M, N + 3, dtype=torch.float32, device=DEV)
    got = acid.acid_linear_forward(_t(a)[:, 3:3 + K], _t(w), None, out=buf[:, 1:1 + N])
    ref = O.linear(a[:, 3:3 + K], w, np.zeros(N, np.float32))
    mag = np.abs(a[:, 3:3 + K]).astype(np.float64) @ np.abs(w).astype(np.float64).T
    assert np.all(np.abs(got.cpu().numpy() - ref) <= (K + 16) * EPS * mag)
    assert not buf[:, 0].any() and not buf[:, 1 + N:].any()


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
