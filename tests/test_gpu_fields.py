"""Field conversion between the stored deviations and the caller's populations: FP32 arrays
take the float-pair arithmetic, FP64 arrays FP64 adds; both name the same values."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

DIMS = [(1, 1, 1), (5, 3, 7), (33, 7, 3), (64, 8, 4)]


def _populations(n, seed):
    rng = np.random.default_rng(seed)
    f = rng.uniform(0.001, 0.4, size=(27, n)) * 10.0 ** rng.uniform(-3, 1, size=(27, n))
    f[0, 0] = 8.0 / 27.0
    f[3, n // 2] = 0.0
    return f.astype(np.float32)


@pytest.mark.parametrize("dims", DIMS)
@pytest.mark.parametrize("storage", ["fp32", "fp16"])
def test_fp32_populations_equal_the_fp64_path(lib, dims, storage):
    """Read: the FP32 value is the rounded FP64 value (half an ulp, 2^-24 relative, with the
    float pair's own 2^-10 of that).  Write: a half-precision deviation is rounded once on
    either path (equal); an FP32 deviation may differ by one ulp (2^-23) at a tie."""
    from paper_1807_02284_gb300 import lbm
    n = dims[0] * dims[1] * dims[2]
    f = _populations(n, 3)
    a, b = lbm.Domain(dims, 0.01, storage=storage), lbm.Domain(dims, 0.01, storage=storage)
    a.write_field(lbm.LBM_FIELD_F, f)
    b.write_field(lbm.LBM_FIELD_F, f.astype(np.float64))
    fa, fb = (d.read_field(lbm.LBM_FIELD_F, lbm.LBM_F64) for d in (a, b))
    w = np.where(np.arange(27) == 0, 8 / 27, np.where(np.arange(27) < 7, 2 / 27,
                 np.where(np.arange(27) < 19, 1 / 54, 1 / 216))).repeat(n)
    if storage == "fp16":
        assert np.array_equal(fa, fb)
    else:
        assert np.all(np.abs(fa - fb) <= 2.0 ** -23 * np.abs(fb - w) + 2.0 ** -52)
    f32 = a.read_field(lbm.LBM_FIELD_F, lbm.LBM_F32).astype(np.float64)
    assert np.all(np.abs(f32 - fa) <= 2.0 ** -24 * (1 + 2.0 ** -10) * np.abs(fa))
    a.close()
    b.close()


@pytest.mark.parametrize("storage", ["fp32", "fp16"])
def test_infinities_and_nan_pass_through(lib, storage):
    from paper_1807_02284_gb300 import lbm
    f = _populations(64, 4)
    f[2, 5], f[9, 6], f[20, 7] = np.inf, -np.inf, np.nan
    d = lbm.Domain((4, 4, 4), 0.01, storage=storage)
    d.write_field(lbm.LBM_FIELD_F, f)
    g = d.read_field(lbm.LBM_FIELD_F, lbm.LBM_F32).reshape(27, 64)
    assert g[2, 5] == np.inf and g[9, 6] == -np.inf and np.isnan(g[20, 7])
    assert np.array_equal(np.isfinite(g), np.isfinite(f))
    d.close()


@pytest.mark.parametrize("dims", DIMS)
@pytest.mark.parametrize("offset", [0, 1])
def test_velocity_and_scalar_copies(lib, dims, offset):
    """Device reads and writes of FP32 fields, 16-byte aligned or not, are exact copies."""
    import torch
    from paper_1807_02284_gb300 import lbm
    n = dims[0] * dims[1] * dims[2]
    d = lbm.Domain(dims, 0.01)
    src = torch.rand(3 * n + offset, device="cuda")[offset:]
    out = torch.zeros(3 * n + offset + 1, device="cuda")
    torch.cuda.synchronize()
    d.write_field(lbm.LBM_FIELD_U, src)
    d.read_field(lbm.LBM_FIELD_U, lbm.LBM_F32, out=out[offset:offset + 3 * n])
    assert torch.equal(out[offset:offset + 3 * n], src) and out[-1] == 0
    d.close()


def _ties(read):
    """Per weight, the values whose sum with (read) or difference from it lies next to a tie of
    FP32, five floats to either side, over magnitudes around the weight; padded to one length."""
    w = np.where(np.arange(27) == 0, 8 / 27, np.where(np.arange(27) < 7, 2 / 27,
                 np.where(np.arange(27) < 19, 1 / 54, 1 / 216)))
    rows = []
    for q in range(27):
        lo = w[q] - np.float64(np.float32(w[q]))
        out = []
        for ex in range(-10, 11):
            u = np.float64(np.spacing(np.float32(w[q] * 2.0 ** ex)))
            for x in list(u * np.arange(-3, 4)) + [w[q] * 2.0 ** ex, -w[q] * 2.0 ** ex]:
                for h in (u / 2, -u / 2, u / 4, -u / 4):
                    v = np.float32(x + h - lo if read else x + h + lo)
                    for side in (np.inf, -np.inf):
                        y = v
                        for _ in range(5):
                            out.append(y)
                            y = np.nextafter(y, np.float32(side))
        rows.append(np.array(out, np.float32))
    return np.stack(rows), w[:, None]


def _domain_of(lbm, n):
    assert n % 8 == 0
    return lbm.Domain((n // 8, 4, 2), 0.01)


def test_fp32_reads_are_the_rounded_fp64_reads(lib):
    """FP32 storage, deviations next to ties of the sum and random ones: the FP32 populations
    are the FP64 ones rounded once, bit for bit."""
    from paper_1807_02284_gb300 import lbm
    dev, w = _ties(True)
    rng = np.random.default_rng(6)
    r = (w * rng.normal(size=(27, 1 << 14)) * 10.0 ** rng.uniform(-8, 1, size=(27, 1 << 14))).astype(np.float32)
    dev = np.concatenate([dev, r], axis=1)
    dev = np.pad(dev, ((0, 0), (0, -dev.shape[1] % 8)))
    d = _domain_of(lbm, dev.shape[1])
    d.write_field(lbm.LBM_FIELD_F, w + dev.astype(np.float64))
    f64 = d.read_field(lbm.LBM_FIELD_F, lbm.LBM_F64)
    f32 = d.read_field(lbm.LBM_FIELD_F, lbm.LBM_F32)
    assert np.array_equal(f32.view(np.uint32), f64.astype(np.float32).view(np.uint32))
    d.close()


def test_fp32_writes_equal_fp64_writes(lib):
    """The same floats handed over as FP32 and as FP64, next to ties of the difference, random and
    special ones: the same stored deviations, bit for bit."""
    from paper_1807_02284_gb300 import lbm
    f, w = _ties(False)
    rng = np.random.default_rng(7)
    r = (w * (1 + rng.normal(size=(27, 1 << 14)) * 10.0 ** rng.uniform(-8, 1, size=(27, 1 << 14)))).astype(np.float32)
    special = np.tile(np.array([np.inf, -np.inf, np.nan, 3e38, -3e38, 1e-45, 0.0, -0.0], np.float32), (27, 1))
    f = np.concatenate([f, r, special, w.astype(np.float32)], axis=1)
    f = np.pad(f, ((0, 0), (0, -f.shape[1] % 8)))
    a, b = _domain_of(lbm, f.shape[1]), _domain_of(lbm, f.shape[1])
    a.write_field(lbm.LBM_FIELD_F, f)
    b.write_field(lbm.LBM_FIELD_F, f.astype(np.float64))
    fa, fb = (d.read_field(lbm.LBM_FIELD_F, lbm.LBM_F64) for d in (a, b))
    assert np.array_equal(fa, fb, equal_nan=True)
    a.close()
    b.close()
