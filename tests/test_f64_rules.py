"""The FP64 step's tile rule, and the reciprocal and roots of its tensor stage."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

import oracle as O

torch = pytest.importorskip("torch")

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)

# tile (width x height) and a size that takes it (Gaussian radius 2 or 3, radius 5)
TILES = {(8, 4): ((52, 59), (40, 43)), (8, 8): ((80, 90), (80, 90)), (16, 16): ((163, 170), (150, 153)),
         (32, 16): ((241, 243), (241, 243)), (32, 20): ((397, 399), (397, 399)), (32, 24): ((449, 447), (449, 447)),
         (32, 28): ((509, 511), (509, 511)), (32, 32): ((346, 353), (346, 353))}


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    from paper_2006_10406_gb300 import build
    out = str(tmp_path_factory.mktemp("probe") / "f64_probe.so")
    subprocess.run([build.nvcc(), *build.ARCH, "-O2", "-std=c++17", "--expt-relaxed-constexpr", "-Xcompiler", "-fPIC", "-shared",
                    "-I", build.INCLUDE, "-I", build.CSRC, os.path.join(HERE, "f64_probe.cu"), "-o", out], check=True)
    return C.CDLL(out)


@pytest.mark.parametrize("tile", list(TILES))
@pytest.mark.parametrize("eed", [0, 1])
@pytest.mark.parametrize("R", [2, 3, 5])
def test_each_tile_has_a_size(probe, tile, eed, R):
    h, w = TILES[tile][R == 5]
    assert probe.f64_probe_tile(R, eed, w, h) == 100 * tile[0] + tile[1]


@pytest.mark.gpu
@pytest.mark.parametrize("method", [0, 1])
@pytest.mark.parametrize("sigma", [0.5, 1.0, 1.5])
def test_step_on_32x32_tiles(probe, method, sigma):
    """Ragged: 346 x 353. Tolerance of one FP64 step as in test_gpu_parity.py."""
    import paper_2006_10406_gb300 as fg
    h, w = TILES[32, 32][0]
    assert probe.f64_probe_tile(int(np.ceil(3 * sigma)), method, w, h) == 3232
    rng = np.random.default_rng(int(10 * sigma))
    ucur = rng.uniform(size=(h, w))
    ucur[:, : w // 3] = 0.5  # zero gradients
    uprev = ucur + 0.01 * rng.normal(size=(h, w))
    mask = (rng.uniform(size=(h, w)) < 0.1).astype(np.uint8)
    tau = 0.05 if method == 0 else 0.25
    ref = O.fsi_step(method, uprev, ucur, mask, 1.4, tau, sigma, 0.03)
    a, b, m = (torch.from_numpy(x).cuda() for x in (uprev, ucur, mask))
    out = torch.empty_like(a)
    (fg.foeed_step if method == 0 else fg.eed_step)(a, b, out, m, 1.4, 0.03, sigma, tau=tau)
    np.testing.assert_allclose(out.cpu().numpy(), ref, rtol=0, atol=1e-12)


@pytest.mark.gpu
def test_reciprocal_and_roots_over_their_range(probe):
    """x in [1e-30, 1e37). The truncation of the second-order step is below 2^-62; on top come the rounding of the
    result (2^-53) and, through h, of y^2 (half of 2^-53 after the factor 1/2) and of y^4 (3/4 of it after 1/4)."""
    rng = np.random.default_rng(1)
    x = np.concatenate([10.0 ** rng.uniform(-30, 37, size=1 << 20), 2.0 ** np.arange(-99, 122), [1e-30, np.nextafter(1e37, 0)]])
    x = x[(x >= 1e-30) & (x < 1e37)]
    xd = torch.from_numpy(x).cuda()
    out = torch.empty(3, len(x), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    assert probe.f64_probe_roots(C.c_void_p(xd.data_ptr()), C.c_void_p(out.data_ptr()), len(x)) == 0
    X = x.astype(np.longdouble)
    root = np.sqrt(X)
    for got, ref, ulps in zip(out.cpu().numpy(), (1 / X, 1 / root, 1 / np.sqrt(root)), (1.0, 1.5, 1.75)):
        err = np.abs(got.astype(np.longdouble) / ref - 1).max()
        assert err <= ulps * 2.0 ** -53 + 2.0 ** -60, float(err * 2.0 ** 53)
