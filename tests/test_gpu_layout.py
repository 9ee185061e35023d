"""Layout conversion between the canonical field and device storage: every entry arrives where it belongs and as
the nearest number of the storage type, for site counts around the kernels' 32-site blocks and for special values.
FP32 storage keeps float32(x) of every entry, so the comparison is exact."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SPECIAL = [0.0, -0.0, 1.0, -1.0, 2.0 ** -126, 2.0 ** -149, -2.0 ** -130, 1e-300, 3.4e38, -1e39, np.inf, -np.inf, np.nan, 1 / 3]


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("Ls", [[(2, 2, 2, 2)], [(2, 2, 2, 4)], [(3, 11, 1 + 1, 2), (2, 2, 2, 3)], [(3, 3, 5, 7), (2, 2, 6, 6), (4, 4, 2, 2)]])
def test_pack_and_unpack_are_exact(tgf, prec, Ls):
    rng = np.random.default_rng(3)
    fields = []
    for L in Ls:
        shape = (L[3], L[2], L[1], L[0], 4, 3, 3)
        f = (rng.standard_normal(shape) + 1j * rng.standard_normal(shape)).astype(np.complex128)
        flat = f.view(np.float64).reshape(-1)
        at = rng.integers(0, flat.size, 200)
        with np.errstate(all="ignore"):
            flat[at] = np.array(SPECIAL)[rng.integers(0, len(SPECIAL), 200)]
        fields.append(f)
    b = tgf.FlowBatch(Ls, prec, any_extents=True)
    b.set_links(fields)
    for f, g in zip(fields, b.get_links()):
        x = f.view(np.float64).reshape(-1)
        with np.errstate(all="ignore"):
            want = x if prec == "fp64" else x.astype(np.float32).astype(np.float64)
        got = g.view(np.float64).reshape(-1)
        assert np.array_equal(np.isnan(got), np.isnan(want))
        ok = ~np.isnan(want)
        assert np.array_equal(got[ok].view(np.int64), want[ok].view(np.int64))
