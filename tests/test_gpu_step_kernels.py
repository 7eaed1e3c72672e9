"""GPU parity of the kernels around the block stack of a step, through short
loops with forced compute and reuse decisions, against the oracle's loop: the
patch gather and scatter in tiles of 32 patches (a partial tile, several
tiles a row, a temporal patch of 2) and element by element (patch vectors of
more than 256 values), and the residual applied and stored in the final
layer's LayerNorm, host-driven and as a graph, in rows of every team width."""

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


SHAPES = [dict(latent_f=2, latent_h=6, latent_w=90), dict(latent_f=4, latent_h=4, latent_w=64, pt=2),
          dict(latent_f=1, latent_h=6, latent_w=10, latent_c=80), dict(latent_f=2, latent_h=4, latent_w=18, latent_c=64)]
FORCED = [None, True, False, False, True, False]


def check_forced_loop(acid, cfg, graph):
    w = S.model_weights(cfg, 5)
    lat = S.latent(cfg, 5)
    model = acid.DeviceModel(cfg, w, DEV)
    c, keep = acid.loop_cfg(cfg, forced=FORCED)
    tl = torch.from_numpy(lat).to(DEV)
    logs = acid.acid_denoise_loop(model, c, tl, None, graph=graph)
    acid.check_device_error()
    ref = O.denoise_loop(cfg, w, lat, None, forced=FORCED)
    assert [bool(l["computed"]) for l in logs] == ref.computed
    got = tl.cpu().numpy()
    if cfg.dtype == "fp32":
        assert np.abs(got - ref.latent).max() <= 1e-4 * np.abs(ref.latent).max()
    else:  # six velocities, each off by the bf16 block's and final layer's 1e-2 at most
        assert np.linalg.norm(got - ref.latent) <= 1e-2 * np.linalg.norm(ref.latent)
    for l, r in zip(logs[1:], ref.records[1:]):
        assert abs(l["signal"] - r.signal) <= 1e-3 * abs(r.signal)


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("d,dtype", [(256, "fp32"), (576, "fp32"), (256, "bf16"), (576, "bf16")])
def test_forced_loop(acid, shape, graph, d, dtype):
    cfg = S.get_config("toy", d=d, heads=d // 64, ffn=128, n_blocks=1, steps=len(FORCED), dtype=dtype, **shape)
    check_forced_loop(acid, cfg, graph)


# teams of three warps (1600: the last lanes empty, 1920: full) and of four (2112,
# 3072), on 920 tokens: more rows than either has teams (912 and 608)
@pytest.mark.parametrize("d", [1600, 1920, 2112, 3072])
@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
def test_forced_loop_wide_rows(acid, d, dtype):
    cfg = S.get_config("toy", d=d, heads=d // 64, ffn=128, n_blocks=1, steps=len(FORCED), dtype=dtype, latent_f=4,
                       latent_h=20, latent_w=46)
    check_forced_loop(acid, cfg, False)
