"""Packing and unpacking at partial blocks of 64 sites, and the numbers that
the integer float-to-double conversion leaves to the conversion instruction."""
import numpy as np
import pytest
import torch

from paper_1311_4521_gb300 import fields as F

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_1311_4521_gb300 import tmhop
    c = tmhop.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("prec,tol", [("f64", 0.0), ("f64x", 1e-14), ("f32", 1e-7), ("f16", 1e-3)])
@pytest.mark.parametrize("vh", [1, 63, 64, 65, 127, 128, 129, 1000])
def test_round_trip(ctx, prec, tol, vh):
    psi = F.gaussian_spinor(vh, 960, vh)
    back = ctx.unpack(ctx.pack(psi, prec), vh, prec).cpu().numpy()
    assert np.abs(back - psi).max() <= tol * np.abs(psi).max()


def test_f32_layout_and_every_kind_of_number(ctx):
    vh = 70
    rng = np.random.default_rng(1)
    x = rng.integers(0, 2 ** 32, size=24 * vh, dtype=np.uint32)
    x[:9] = [0, 0x80000000, 1, 0x807fffff, 0x00800000, 0x7f7fffff, 0x7f800000, 0xff800000, 0x7fc00000]
    f = x.view(np.float32)
    f = np.where(np.isnan(f) & (np.arange(f.size) != 8), np.float32(1), f)
    got = ctx.unpack(torch.from_numpy(f.copy()).cuda().view(torch.uint8), vh, "f32").cpu().numpy().view(np.float64).reshape(vh, 24)
    want = f.reshape(6, vh, 4).transpose(1, 0, 2).reshape(vh, 24).astype(np.float64)   # 6 arrays of float4
    assert np.array_equal(got, want, equal_nan=True)
    assert np.array_equal(np.signbit(got[want == 0]), np.signbit(want[want == 0]))
    back = ctx.pack(torch.from_numpy(got.view(np.complex128).reshape(vh, 4, 3)), "f32").cpu().numpy().view(np.float32)
    assert np.array_equal(back, f, equal_nan=True)
