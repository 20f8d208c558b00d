"""osog_sensor_noise against the FP64 oracle (same Philox streams, same
Poisson decisions), reproducibility independent of the launch, in-place
use and argument checks."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _img(n, seed=0):
    rng = np.random.default_rng(seed)
    x = rng.uniform(0.0, 2.0, n).astype(np.float32)
    x[::97] = -0.1  # clipped to zero photons
    x[::89] = 0.0
    return x


@pytest.mark.parametrize("g,sigma", [(0.5, 0.0), (20.0, 3.0), (5000.0, 2.0), (3e6, 40.0)])
def test_matches_the_oracle(g, sigma):
    from paper_2606_21381_gb300.noise import sensor_noise
    x = _img(512 * 512)
    want = oracle.sensor_noise(x, g, sigma, 12345)
    got = sensor_noise(torch.from_numpy(x).cuda(), g, sigma, 12345).cpu().numpy()
    np.testing.assert_allclose(got, want, rtol=2e-7, atol=1e-9)


def test_draw_depends_only_on_seed_and_index():
    from paper_2606_21381_gb300.noise import sensor_noise
    x = torch.from_numpy(_img(3 * 2048 * 2048 + 17, 1)).cuda()
    a = sensor_noise(x, 1000.0, 1.5, 7)
    b = sensor_noise(x, 1000.0, 1.5, 7)
    assert torch.equal(a, b)
    part = sensor_noise(x[:100_003].contiguous(), 1000.0, 1.5, 7)
    assert torch.equal(part, a[:100_003])
    assert not torch.equal(sensor_noise(x, 1000.0, 1.5, 8), a)
    idx = np.array([0, 5, 12_582_911, 12_582_928])
    xs = x.cpu().numpy()
    for i in idx:
        lam = 1000.0 * max(float(xs[i]), 0.0)
        want = (oracle.poisson(lam, 7, int(i)) + 1.5 * oracle.normal(7, int(i))) / 1000.0
        assert abs(float(a[i]) - want) <= 2e-7 * abs(want) + 1e-9


def test_in_place_and_argument_checks():
    from paper_2606_21381_gb300._lib import OsogError
    from paper_2606_21381_gb300.noise import sensor_noise
    x = torch.from_numpy(_img(10_000, 2)).cuda()
    want = sensor_noise(x, 50.0, 1.0, 3)
    y = x.clone()
    sensor_noise(y, 50.0, 1.0, 3, out=y)
    assert torch.equal(y, want)
    for g, s in ((0.0, 1.0), (-1.0, 1.0), (10.0, -1.0), (10.0, float("nan"))):
        with pytest.raises(OsogError):
            sensor_noise(x, g, s, 3)


# both sides of every boundary of the FP32 draw: rates at and around 10 and
# 2^22, gains and read noises outside its range, images that are dark, far too
# bright or not finite
@pytest.mark.parametrize("g,sigma,level", [
    (10.0, 1.0, 1.0), (9.999999, 0.5, 1.0), (10.0 / 3.0, 0.0, 3.0), (4194304.0, 2.0, 1.0),
    (1e-7, 1.0, 2e8), (100.0, 1e-7, 1.0), (100.0, 2e6, 1.0), (50.0, 1.0, 0.0)])
def test_boundaries_of_the_fp32_draw(g, sigma, level):
    from paper_2606_21381_gb300.noise import sensor_noise
    x = np.full(20_011, level, dtype=np.float32)
    x[1::3] = np.nextafter(np.float32(level), np.float32(0.0))
    x[2::3] = np.nextafter(np.float32(level), np.float32(4.0 * level + 1.0))
    x[::1009] = 0.0
    x[5] = np.nan  # no photons, like every value that is not above zero
    want = oracle.sensor_noise(np.nan_to_num(x), g, sigma, 99)
    got = sensor_noise(torch.from_numpy(x).cuda(), g, sigma, 99).cpu().numpy()
    np.testing.assert_allclose(got, want, rtol=2e-7, atol=1e-9)


# tiles of one to four elements a thread, whole and ragged, up to several tiles a CTA
@pytest.mark.parametrize("n", [1, 31, 255, 257, 1023, 155_648, 155_649, 311_297, 466_945, 622_593, 700_001])
@pytest.mark.parametrize("g", [3.0, 1000.0])
def test_draws_do_not_depend_on_the_size_of_the_launch(n, g):
    from paper_2606_21381_gb300.noise import sensor_noise
    x = torch.rand(1_400_000, generator=torch.Generator().manual_seed(n)).cuda() * 4.0
    want = sensor_noise(x, g, 1.5, 11)
    assert torch.equal(sensor_noise(x[:n], g, 1.5, 11), want[:n])


@pytest.mark.parametrize("g,run", [(4e6, 1), (4e6, 64), (1e-7, 64), (1e8, 64)])
def test_warps_in_and_out_of_the_fp32_draws_range(g, run):
    # runs of pixels brighter and darker than 2^22 photons, of one lane and of two
    # warps, and gains that no pixel's or every pixel's FP32 draw takes
    from paper_2606_21381_gb300.noise import sensor_noise
    x = np.where((np.arange(5000) // run) % 2 == 0, 0.5, 1.5).astype(np.float32)
    x[17::301] = 0.0
    want = oracle.sensor_noise(x, g, 2.0, 7)
    got = sensor_noise(torch.from_numpy(x).cuda(), g, 2.0, 7).cpu().numpy()
    np.testing.assert_allclose(got, want, rtol=2e-7, atol=1e-9)
