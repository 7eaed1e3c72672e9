"""GPU parity of the SM-pair GEMM at every tile width its dispatch can choose,
with ragged rows, columns and K, of residual rows that overlap, and of
dual-stream layers whose text and video rows share a launch."""

import numpy as np
import pytest

import acid_synth as S
import oracle as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

DEV = "cuda"


@pytest.fixture(scope="module")
def acid():
    import __graft_entry__ as g

    g.build()
    from paper_2607_12358_gb300 import acid as a

    return a


def _bf(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).to(DEV, torch.bfloat16)


def _f32(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).to(DEV)


def _tol(a, w, extra, K, out_fp32):
    """fp32 accumulation of K products (K 2^-24 of the terms' magnitudes), then
    for bf16 output one rounding (2^-9 relative, 2^-8 with its neighbours)."""
    mag = np.abs(a).astype(np.float64) @ np.abs(w).astype(np.float64).T + extra
    return mag * (K + 16) * 2.0 ** -24 * 4, 0.0 if out_fp32 else 2.0 ** -8


# on 76 SM pairs these shapes get tiles of 32, 64, 96, 128, 160, 192, 224 and
# 256 columns, each with a partial last column tile, row tile and k-block
@pytest.mark.parametrize("M,K,N", [(1, 72, 1056), (130, 72, 2464), (513, 72, 4064), (1000, 72, 3680), (1290, 72, 3712),
                                   (1290, 200, 4064), (2000, 72, 3680), (4300, 712, 992)])
@pytest.mark.parametrize("epi,fp32", [("bias", True), ("gelu", False), ("gated_res", True), ("gated_res", False),
                                      ("res", True), ("res", False)])
def test_pair_tile_widths(acid, M, K, N, epi, fp32):
    rng = np.random.default_rng(M + 3 * K + 5 * N)
    a = S.round_to_bf16(rng.normal(size=(M, K)).astype(np.float32))
    w = S.round_to_bf16((0.1 * rng.normal(size=(N, K))).astype(np.float32))
    b, g = rng.normal(size=N).astype(np.float32), rng.normal(size=N).astype(np.float32)
    r = rng.normal(size=(M, N)).astype(np.float32)
    if not fp32:
        r = S.round_to_bf16(r)
    res = (_f32(r) if fp32 else _bf(r)) if epi in ("gated_res", "res") else None
    got = acid.acid_linear_forward(_bf(a), _bf(w), _f32(b), epilogue=epi, gate=_f32(g), residual=res, out=res,
                                   out_fp32=fp32).float().cpu().numpy()
    acc = O.linear(a, w, b)
    ref = {"bias": acc, "gelu": O.gelu_tanh(acc), "gated_res": r + g * acc, "res": r + acc}[epi]
    absolute, rel = _tol(a, w, np.abs(b) + np.abs(r), K, fp32)
    if epi == "gated_res":
        absolute = absolute * np.maximum(1.0, np.abs(g))
    # GELU adds the error of tanh.approx: 2^-11 of |x| / 2
    slack = 2.0 ** -11 * np.abs(acc) if epi == "gelu" else 0.0
    assert np.all(np.abs(got - ref) <= absolute + slack + rel * np.abs(ref))


@pytest.mark.parametrize("ldr", [0, 8])
@pytest.mark.parametrize("fp32", [True, False])
def test_residual_rows_that_overlap(acid, ldr, fp32):
    """A residual with a row stride below its width: one row added to every
    output row (stride 0), and rows 8 elements apart."""
    M, K, N = 300, 72, 160
    rng = np.random.default_rng(11)
    a = S.round_to_bf16(rng.normal(size=(M, K)).astype(np.float32))
    w = S.round_to_bf16((0.1 * rng.normal(size=(N, K))).astype(np.float32))
    flat = S.round_to_bf16(rng.normal(size=N + M * 8).astype(np.float32))
    r = np.stack([flat[i * ldr:i * ldr + N] for i in range(M)])
    dev = _f32(flat) if fp32 else _bf(flat)
    res = torch.as_strided(dev, (M, N), (ldr, 1))
    got = acid.acid_linear_forward(_bf(a), _bf(w), None, epilogue="res", residual=res, out_fp32=fp32)
    ref = r + O.linear(a, w, np.zeros(N, np.float32))
    absolute, rel = _tol(a, w, np.abs(r), K, fp32)
    assert np.all(np.abs(got.float().cpu().numpy() - ref) <= absolute + rel * np.abs(ref))


@pytest.mark.parametrize("n_text", [0, 1, 255, 256, 300])
def test_dual_stream_rows_share_a_launch(acid, n_text):
    """Text rows of less than, exactly and more than one 256-row tile, and
    none: each stream keeps its own weights, bias, modulation and rows."""
    cfg = S.get_config("hv", d=256, heads=2, ffn=1024, n_text=n_text, latent_f=3, latent_h=16, latent_w=22)
    w = S.block_weights(cfg, 0, seed=4, block_type="hv_dual", q_scale=4.0)
    x = S.hidden(cfg, cfg.n_video + n_text, seed=n_text)
    temb = S.temb_vector(cfg, seed=4)
    blk = acid.DeviceBlock.upload(w, "hv_dual", torch.bfloat16, DEV)
    got = acid.acid_dit_block_forward(acid.block_desc(cfg, "hv_dual"), _bf(x), _f32(temb), blk).float().cpu().numpy()
    acid.check_device_error()
    mt, mv = O.block_modulation(temb, w["txt.mod"]), O.block_modulation(temb, w["vid.mod"])
    if n_text:
        yt, yv = O.hv_dual_block(x[:n_text], x[n_text:], mt, mv, w, cfg.grid, cfg.heads)
    else:  # the video stream alone: self-attention and FFN with its weights
        vid = {k[4:]: v for k, v in w.items() if k.startswith("vid.")}
        yt, yv = x[:0], O.wan_block(x, mv, vid, cfg.grid, cfg.heads)
    # the block tolerance of the bf16 path, for each stream by itself
    for g, r in ((got[:n_text], yt), (got[n_text:], yv)):
        if r.size:
            assert np.linalg.norm(g - r) <= 1e-2 * np.linalg.norm(r) and np.abs(g - r).max() <= 5e-2
