"""The density moment at the edges of its sums: planes and slices of every
alignment and remainder, one block a plane and several slices, both block
sizes, and values whose alignment to a common exponent is at its limits."""
import numpy as np
import pytest

from paper_2303_14119_gb300 import fk

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    fk.load()
    return torch


def moment(torch, f, offset=0):
    """n_e of f [nx][nv1][nv2] from device memory `offset` values past an aligned address."""
    buf = torch.zeros(f.size + offset, dtype=torch.float64, device="cuda")
    buf[offset:] = torch.from_numpy(f.reshape(-1)).cuda()
    n_e = torch.full((f.shape[0],), float("nan"), dtype=torch.float64, device="cuda")
    fk.fk_density_moment_noalloc(buf.data_ptr() + 8 * offset, *f.shape, 1.0, 1.0, n_e.data_ptr(),
                                 torch.cuda.current_stream().cuda_stream or None)
    torch.cuda.synchronize()
    return n_e.cpu().numpy()


# one value, less than a group, a group's edge, several groups; slices (nx < 64)
# and whole planes; 256 and 512 threads
@pytest.mark.parametrize("shape", [(1, 1, 1), (3, 1, 7), (5, 16, 255), (63, 4, 1025), (64, 3, 5),
                                   (70, 64, 65), (64, 128, 129), (2, 517, 1031)])
@pytest.mark.parametrize("offset", [0, 1])
def test_sums_of_every_alignment(torch, shape, offset):
    rng = np.random.default_rng(shape[0] + offset)
    f = rng.uniform(size=shape) * 10.0 ** rng.uniform(-30, 5, size=shape)
    ref = f.astype(np.longdouble).sum(axis=(1, 2)).astype(np.float64)
    got = moment(torch, f, offset)
    # rounded once a group and block, positive terms: a few ulp
    assert np.abs(got - ref).max() <= 1e-15 * np.abs(ref).max()


@pytest.mark.parametrize("scale", [1.0, 2.0 ** -1000, 5e-324, 2.0 ** 1000])
def test_sums_at_the_ends_of_the_range(torch, scale):
    rng = np.random.default_rng(3)
    f = rng.integers(1, 1000, size=(66, 9, 11)).astype(np.float64) * scale
    assert np.array_equal(moment(torch, f), f.sum(axis=(1, 2)))  # whole numbers of scale: exact


def test_negative_and_non_finite_values(torch):
    f = np.ones((65, 8, 9))
    f[1, 2, 3] = -5.0
    f[2, 1, 1] = np.inf
    f[3, 0, 0] = np.nan
    f[4] = 0.0
    f[5, 4, 4] = -0.0
    got = moment(torch, f)
    assert got[0] == 72.0 and got[1] == 66.0 and got[4] == 0.0 and got[5] == 71.0
    assert np.isposinf(got[2]) and np.isnan(got[3]) and np.all(got[6:] == 72.0)


# small planes whole and larger ones in slices below 64 planes, large planes in four
@pytest.mark.parametrize("shape", [(2, 128, 128), (2, 113, 146), (64, 512, 512), (65, 513, 513),
                                   (303, 512, 512), (304, 512, 512)])
def test_sums_on_either_side_of_the_slicing_rule(torch, shape):
    gen = torch.Generator(device="cuda").manual_seed(shape[0])
    f = torch.rand(shape, generator=gen, dtype=torch.float64, device="cuda")
    n_e = torch.empty(shape[0], dtype=torch.float64, device="cuda")
    fk.fk_density_moment_noalloc(f.data_ptr(), *shape, 1.0, 1.0, n_e.data_ptr(),
                                 torch.cuda.current_stream().cuda_stream or None)
    # multiples of 2^-53 below 1: whole sums below 2^64 as two halves
    hi = torch.floor(f * 2.0 ** 26).to(torch.int64)
    lo = (f * 2.0 ** 26 - hi) * 2.0 ** 27
    ref = (hi.sum((1, 2)).double() + lo.to(torch.int64).sum((1, 2)).double() * 2.0 ** -27) * 2.0 ** -26
    assert ((n_e - ref).abs() <= 1e-15 * ref).all()


def test_few_large_planes_take_no_longer_than_many_small_ones(torch):
    """The same 0.5 GB as 64 planes and as 1024: 87 and 82 us (166 with 64 blocks
    on 152 SMs)."""
    def best(shape):
        f = torch.rand(shape, dtype=torch.float64, device="cuda")
        n_e = torch.empty(shape[0], dtype=torch.float64, device="cuda")
        times = []
        for _ in range(8):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            for _ in range(10):
                fk.fk_density_moment_noalloc(f.data_ptr(), *shape, 1.0, 1.0, n_e.data_ptr(),
                                             torch.cuda.current_stream().cuda_stream or None)
            e1.record()
            torch.cuda.synchronize()
            times.append(e0.elapsed_time(e1))
        return min(times)
    assert best((64, 1024, 1024)) < 1.5 * best((1024, 256, 256))
