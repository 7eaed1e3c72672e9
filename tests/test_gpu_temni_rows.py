"""GPU parity of the TEMNI drift where several warps share a row (more than
1536 columns), at the edges of its column split and with fewer and more rows
than row groups, against the CPU oracle's definition."""

import numpy as np
import pytest

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


# 1544 and 1920: the last of four vectors per lane only partly filled; 2048 and
# 3072: every lane full; 2056 and 3064 on either side.  Three or four groups a CTA
# on 152 CTAs: 2500 rows give every group several, 5 rows leave most without one
@pytest.mark.parametrize("d", [1544, 1920, 2048, 2056, 3064, 3072])
@pytest.mark.parametrize("rows", [1, 5, 457, 2500])
def test_temni_drift_wide_rows(acid, rows, d):
    rng = np.random.default_rng(rows + d)
    hp = (0.5 + rng.normal(size=(rows, d))).astype(np.float32)
    hc = (hp + 0.05 * rng.normal(size=(rows, d))).astype(np.float32)
    mp, mc = rng.normal(size=2 * d).astype(np.float32), rng.normal(size=2 * d).astype(np.float32)
    t = lambda a: torch.from_numpy(a).to(DEV)  # noqa: E731
    rel, sums = acid.acid_temni_drift(t(hp), t(hc), t(mp), t(mc))
    acid.check_device_error()
    prev, cur = (O.modulate(O.layer_norm(h), m[:d], m[d:]) for h, m in ((hp, mp), (hc, mc)))
    num, den = np.abs(cur - prev).sum(), np.abs(prev).sum()
    # every term carries a few fp32 roundings, mostly of either sign: 1e-5 is
    # a hundred times their relative size
    assert abs(sums[0].item() - num) <= 1e-5 * num and abs(sums[1].item() - den) <= 1e-5 * den
    assert abs(rel.item() - num / den) <= 2e-5 * num / den
    again, _ = acid.acid_temni_drift(t(hp), t(hc), t(mp), t(mc))
    assert again.item() == rel.item()
