"""GPU parity of the two LayerNorm kernels (one warp per row up to 512 columns;
persistent teams of two, three or four warps on bulk copies) on both sides of
the widths between them, with rows that do not fill the last lanes, ragged
last rounds, rings of two and four rows and every pair of types, and of the
joint blocks' split between text and video modulation."""

import numpy as np
import pytest

import acid_synth as S
import oracle as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

DEV = "cuda"
DT = {"bf16": torch.bfloat16, "fp32": torch.float32}


@pytest.fixture(scope="module")
def acid():
    import __graft_entry__ as g

    g.build()
    from paper_2607_12358_gb300 import acid as a

    return a


# 512, 1536 and 1920 columns are the widest of their kernel; 1216, 912 and 608
# rows give each team of two, three and four warps one; the last two sizes lie on
# both sides of 160 MB in bf16
@pytest.mark.parametrize("rows,d", [(1, 8), (5, 264), (12159, 520), (12160, 520), (12161, 1536), (12300, 1544),
                                    (12200, 2048), (12170, 3072), (12163, 512), (777, 1928), (300, 3064), (1217, 1528),
                                    (913, 1920), (4000, 1912), (609, 3072), (13020, 3072), (13024, 3072)])
@pytest.mark.parametrize("tin,tout", [("bf16", "bf16"), ("bf16", "fp32"), ("fp32", "bf16"), ("fp32", "fp32")])
@pytest.mark.parametrize("mod", [True, False])
def test_layernorm_kernels(acid, rows, d, tin, tout, mod):
    rng = np.random.default_rng(rows + d)
    x = (rng.normal(size=(rows, d)) * 2 + 3).astype(np.float32)  # a mean well away from zero
    if tin == "bf16":
        x = S.round_to_bf16(x)
    sh, sc = (rng.normal(size=d).astype(np.float32) for _ in range(2))
    dev = torch.from_numpy(x).to(DEV, DT[tin])
    t = [torch.from_numpy(v).to(DEV) if mod else None for v in (sh, sc)]
    got = acid.acid_layernorm_mod(dev, *t, out_dtype=DT[tout]).float().cpu().numpy()
    acid.check_device_error()
    x64 = x.astype(np.float64)
    n = (x64 - x64.mean(1, keepdims=True)) / np.sqrt(x64.var(1, keepdims=True) + 1e-6)
    ref = n * (1.0 + sc) + sh if mod else n
    # mean and variance each add up to d roundings of 2^-24, relative to |x|
    # about 5 at a spread of 2; bf16 output rounds once more
    tol = (np.abs(n) + 3.0) * (1.0 + np.abs(sc) if mod else 1.0) * (16 + np.sqrt(d)) * 2.0 ** -24 + np.abs(ref) * 2.0 ** -22
    if tout == "bf16":
        tol = tol + np.abs(ref) * 2.0 ** -8
    assert np.all(np.abs(got - ref) <= tol)


@pytest.mark.parametrize("n_text,f", [(37, 3), (226, 48)])
def test_joint_block_streams_keep_their_modulation(acid, n_text, f):
    """A joint block of 829 rows (a row a team) and of 12898 rows
    (several), checked by the oracle on the rows around the split, where
    the text stream's modulation ends, and at both ends."""
    cfg = S.get_config("cog", d=576, heads=9, ffn=128, n_text=n_text, latent_f=f, latent_h=16, latent_w=66)
    w = S.block_weights(cfg, 0, seed=3)
    rows = cfg.n_video + n_text
    x = S.hidden(cfg, rows, seed=3)
    temb = S.temb_vector(cfg, seed=3)
    blk = acid.DeviceBlock.upload(w, "cog", torch.bfloat16, DEV)
    got = acid.acid_dit_block_forward(acid.block_desc(cfg, "cog"), torch.from_numpy(x).to(DEV, torch.bfloat16),
                                      torch.from_numpy(temb).to(DEV), blk).float().cpu().numpy()
    acid.check_device_error()
    at = np.array([0, 1, n_text - 2, n_text - 1, n_text, n_text + 1, rows - 1])
    ref = O.cog_block(x, O.block_modulation(temb, w["mod"]), w, cfg.grid, cfg.heads, n_text, rows=at)
    for r, v in zip(at, ref):
        assert np.linalg.norm(got[r] - v) <= 1e-2 * np.linalg.norm(v), r
