"""Kernels chosen by size, type, alignment or model variant, each against the FP64 oracle
at the edges of its tiles and of its dispatch rule.

Tolerances: one FP64 step 1e-12, one FP32 step 2e-5 (float rounding of |tau P u| <=
tau * 32 * max|u|), as in test_gpu_parity.py."""
import ctypes as C
import threading

import numpy as np
import pytest

import oracle as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - the marker deselects these on CPU
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2006_10406_gb300 as fg  # noqa: E402

DEV = torch.device("cuda", 0)


def _dev(a, dtype):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV, dtype)


def _step(method, uprev, ucur, mask, alpha, lam, sigma, dtype, pitch=None, **kw):
    """One step on images of the given row pitch; the result as float64."""
    h, w = ucur.shape
    pitch = pitch or w

    def place(a, dt):
        t = torch.zeros(h * pitch + 64, device=DEV, dtype=dt)[:h * pitch].as_strided((h, w), (pitch, 1))
        t.copy_(_dev(a, dt))
        return t

    a, b, m = place(uprev, dtype), place(ucur, dtype), place(mask, torch.uint8)
    out = place(np.zeros((h, w)), dtype)
    (fg.foeed_step if method == 0 else fg.eed_step)(a, b, out, m, alpha, lam, sigma, **kw)
    return out.cpu().numpy().astype(np.float64)


@pytest.mark.parametrize("shape", [(1, 9), (15, 63), (17, 65), (16, 64), (33, 130)])
@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("offset", [0, 1])
def test_tensor_field_tiles_and_unaligned_coefficients(shape, dtype, offset):
    """Edges of the 64 (FP64: 32) x 16 tiles; offset 1: coefficients off a 16-byte boundary."""
    rng = np.random.default_rng(shape[0] + 100 * shape[1])
    h, w = shape
    u, d = rng.uniform(size=shape), rng.normal(size=(h, w, 16))
    ud = _dev(u, dtype)
    buf = torch.zeros(h * w * 16 + 4, device=DEV, dtype=dtype)
    buf[offset:offset + h * w * 16] = _dev(d.ravel(), dtype)
    out = torch.empty_like(ud)
    code = fg.F64 if dtype == torch.float64 else fg.F32
    ptr = buf.data_ptr() + offset * buf.element_size()
    assert fg.lib().foeed_apply_tensor_field(C.c_void_p(ud.data_ptr()), C.c_void_p(ptr), C.c_void_p(out.data_ptr()), w, h,
                                             w, code, C.c_void_p(torch.cuda.current_stream().cuda_stream)) == 0
    ref = O.apply_P_field(u, d.reshape(h, w, 2, 2, 2, 2))
    atol = 1e-12 if dtype == torch.float64 else 1e-4 * max(1.0, np.abs(ref).max())
    np.testing.assert_allclose(out.cpu().numpy(), ref, rtol=0, atol=atol)


@pytest.mark.parametrize("method", [0, 1])
@pytest.mark.parametrize("g,mu3", [(0, 1), (0, 2), (1, 0), (1, 1), (2, 0), (2, 2)])
@pytest.mark.parametrize("sigma", [0.0, 0.5, 1.0, 1.5, 2.0])
def test_variants_on_both_kernels(method, g, mu3, sigma):
    """Diffusivities and mu3 choices on the register-blocked kernel (pitch a multiple of 4, both tile
    heights, a flat region with zero gradients) and on the generic one (odd pitch)."""
    if method == 1 and g == 0:
        pytest.skip("EED has no mu3: the default kernel")
    rng = np.random.default_rng(7 * g + mu3)
    shape = (37, 70)
    ucur = rng.uniform(size=shape).astype(np.float32).astype(np.float64)
    ucur[:, 40:] = 0.25
    uprev = (ucur + 0.01 * rng.normal(size=shape)).astype(np.float32).astype(np.float64)
    mask = (rng.uniform(size=shape) < 0.1).astype(np.uint8)
    tau, lam = (0.05 if method == 0 else 0.25), 0.05
    ref = O.fsi_step(method, uprev, ucur, mask, 1.5, tau, sigma, lam, g, mu3)
    got = {}
    for name, pitch, policy in (("h16", 72, "h16"), ("h32", 72, "h32"), ("generic", 71, "auto")):
        fg.set_tile_policy(policy)
        try:
            got[name] = _step(method, uprev, ucur, mask, 1.5, lam, sigma, torch.float32, pitch, tau=tau, diffusivity=g,
                              mu3_mode=mu3)
        finally:
            fg.set_tile_policy("auto")
        np.testing.assert_allclose(got[name], ref, rtol=0, atol=2e-5)
        np.testing.assert_array_equal(got[name][mask != 0], ucur[mask != 0])
    np.testing.assert_array_equal(got["h16"], got["h32"])


@pytest.mark.parametrize("g", [3, 4])
@pytest.mark.parametrize("method", [0, 1])
def test_unbounded_diffusivities(method, g):
    """Aubert and Geman-Reynolds g (EED: register-blocked kernel; FOEED: generic), whose T at a zero
    gradient depends on the direction taken there."""
    rng = np.random.default_rng(g)
    shape = (20, 68)
    ucur = rng.uniform(size=shape).astype(np.float32).astype(np.float64)
    ucur[:, 30:] = 0.5
    ucur[12, 50] = 0.75
    mask = np.zeros(shape, dtype=np.uint8)
    lam, tau = 1.3, 0.05  # g <= 2 / lam^2 stays of order one
    ref = O.fsi_step(method, ucur, ucur, mask, 1.5, tau, 0.0, lam, g, 0)
    got = _step(method, ucur, ucur, mask, 1.5, lam, 0.0, torch.float32, tau=tau, diffusivity=g)
    np.testing.assert_allclose(got, ref, rtol=0, atol=2e-5)


@pytest.mark.parametrize("method", [0, 1])
# the tile the size rule takes: 8 x 4, 8 x 8, 16 x 16, 32 x 16, 32 x 32, ragged
@pytest.mark.parametrize("shape", [(61, 67), (95, 97), (190, 193), (257, 255), (383, 390)])
@pytest.mark.parametrize("sigma", [0.5, 1.5])
def test_f64_tile_shapes(method, shape, sigma):
    rng = np.random.default_rng(shape[0])
    ucur = rng.uniform(size=shape)
    ucur[:, : shape[1] // 3] = 0.5  # zero gradients
    uprev = ucur + 0.01 * rng.normal(size=shape)
    mask = (rng.uniform(size=shape) < 0.1).astype(np.uint8)
    tau = 0.05 if method == 0 else 0.25
    ref = O.fsi_step(method, uprev, ucur, mask, 1.4, tau, sigma, 0.03)
    got = _step(method, uprev, ucur, mask, 1.4, 0.03, sigma, torch.float64, tau=tau)
    np.testing.assert_allclose(got, ref, rtol=0, atol=1e-12)
    np.testing.assert_array_equal(got[mask != 0], ucur[mask != 0])


@pytest.mark.parametrize("method", [0, 1])
# 32 x 20 (two sizes), 32 x 24, 32 x 28 tiles
@pytest.mark.parametrize("shape", [(397, 399), (599, 605), (449, 447), (509, 511)])
@pytest.mark.parametrize("sigma", [0.5, 1.5])
def test_f64_tile_heights_that_fill_the_last_wave(method, shape, sigma):
    rng = np.random.default_rng(shape[0])
    ucur = rng.uniform(size=shape)
    uprev = ucur + 0.01 * rng.normal(size=shape)
    mask = (rng.uniform(size=shape) < 0.1).astype(np.uint8)
    tau = 0.05 if method == 0 else 0.25
    ref = O.fsi_step(method, uprev, ucur, mask, 1.4, tau, sigma, 0.03)
    got = _step(method, uprev, ucur, mask, 1.4, 0.03, sigma, torch.float64, tau=tau)
    np.testing.assert_allclose(got, ref, rtol=0, atol=1e-12)


@pytest.mark.parametrize("method", [0, 1])
@pytest.mark.parametrize("scale", [1e-18, 1e-14, 1e16, 1e20, 1e60])
def test_f64_gradients_beyond_the_fp32_seed_range(method, scale):
    """Images scaled so that squared gradients leave (and straddle) the range of the FP32 seeds."""
    rng = np.random.default_rng(3)
    shape = (24, 40)
    ucur = rng.uniform(size=shape) * scale
    ucur[:, 20:] *= 1e-3
    mask = np.zeros(shape, dtype=np.uint8)
    tau = 0.05 if method == 0 else 0.25
    for lam in (0.03 * scale, 0.03):
        ref = O.fsi_step(method, ucur, ucur, mask, 1.4, tau, 1.0, lam)
        got = _step(method, ucur, ucur, mask, 1.4, lam, 1.0, torch.float64, tau=tau)
        np.testing.assert_allclose(got, ref, rtol=0, atol=1e-12 * scale)


# --------------------------------------------------------------------------
# small images: all steps in cooperative launches, against one launch per step


def _image(h, w, seed):
    rng = np.random.default_rng(seed)
    img = np.clip(0.5 + 0.3 * np.sin(np.arange(w) / 9.0)[None] * np.cos(np.arange(h) / 7.0)[:, None]
                  + 0.05 * rng.normal(size=(h, w)), 0, 1)
    return _dev(img, torch.float32), _dev(rng.uniform(size=(h, w)) < 0.08, torch.uint8)


def _both(method, f, m, lam, sigma, n, cycles, **kw):
    """(result, report) of the cooperative solve and of the step-by-step one (fixed tile policy)."""
    solve = fg.foeed_inpaint if method == 0 else fg.eed_inpaint
    a = solve(f, m, lam, sigma, n, cycles, raise_on_status=False, **kw)
    fg.set_tile_policy("h16")
    try:
        return a, solve(f, m, lam, sigma, n, cycles, raise_on_status=False, **kw)
    finally:
        fg.set_tile_policy("auto")


def _same(a, b):
    assert torch.equal(a[0], b[0])
    assert (a[1].status, a[1].cycles_run, a[1].converged) == (b[1].status, b[1].cycles_run, b[1].converged)
    assert a[1].last_rel_change == pytest.approx(b[1].last_rel_change, rel=1e-12)  # an FP64 sum in another order


@pytest.mark.parametrize("method", [0, 1])
# one tile; partial tiles one pixel wide or high; a side of the smallest size; 64 x 8 tiles, 64 x 16
# tiles with two and with up to four per SM
@pytest.mark.parametrize("shape", [(16, 16), (17, 65), (33, 129), (127, 64), (130, 1000), (250, 511), (512, 515), (700, 701)])
@pytest.mark.parametrize("sigma", [0.0, 0.5, 1.0, 2.0])
def test_cooperative_solve_is_the_stepwise_solve(method, shape, sigma):
    f, m = _image(*shape, seed=shape[0])
    _same(*_both(method, f, m, 0.05, sigma, 7, 4))


@pytest.mark.parametrize("method,kw", [(0, {}), (1, {}), (0, dict(dtype="f32_f64u"))])
@pytest.mark.parametrize("shape", [(705, 705), (17, 19400), (1203, 511)])
def test_cooperative_solve_of_over_512_tiles(method, kw, shape):
    """More tiles than half of the solve's reduction partials."""
    f, m = _image(*shape, seed=2)
    _same(*_both(method, f, m, 0.05, 1.0, 7, 4, **kw))


@pytest.mark.parametrize("method,kw", [(0, {}), (1, {}), (0, dict(dtype="f32_f64u")), (0, dict(diffusivity=1, mu3_mode=1))])
# 64 x 24 tiles: three per SM; one row and one column of pixels over; flat; four per SM; one tile row too many
@pytest.mark.parametrize("shape", [(625, 1000), (625, 1025), (25, 19400), (720, 1280), (912, 1024), (913, 1024)])
@pytest.mark.parametrize("sigma", [0.5, 1.0, 1.5, 2.0])
def test_cooperative_solve_on_24_high_tiles(method, kw, shape, sigma):
    f, m = _image(*shape, seed=4)
    _same(*_both(method, f, m, 0.05, sigma, 7, 4, **kw))


@pytest.mark.parametrize("kw", [dict(dtype="f32_f64u"), dict(diffusivity=1, mu3_mode=1), dict(diffusivity=2)])
@pytest.mark.parametrize("shape", [(61, 90), (300, 400), (600, 600)])
def test_cooperative_solve_of_each_model(kw, shape):
    f, m = _image(*shape, seed=3)
    _same(*_both(0, f, m, 0.05, 1.5, 5, 3, **kw))


@pytest.mark.parametrize("n,cycles", [(2, 1), (2, 9), (3, 4), (128, 3), (100, 85), (129, 2)])
def test_cooperative_cycle_counts(n, cycles):
    """Shortest and longest cycles, odd and even counts, several launches (100 x 85 steps), one step too many."""
    f, m = _image(40, 150, seed=n)
    _same(*_both(0, f, m, 0.05, 1.0, n, cycles))


@pytest.mark.parametrize("n", [2, 3, 30])
@pytest.mark.parametrize("tol", [1e-2, 1e-3, 1e-4])
def test_cooperative_solve_stops_at_the_same_cycle(n, tol):
    f, m = _image(100, 130, seed=n)
    for method in (0, 1):
        _same(*_both(method, f, m, 0.05, 1.0, n, 60, tol=tol))


def test_cooperative_solve_stops_where_it_diverges():
    f, m = _image(64, 100, seed=1)
    a, b = _both(0, f, m, 0.05, 1.0, 20, 50, tau=0.4)
    assert a[1].status == 4 and a[1].cycles_run == b[1].cycles_run and a[1].status == b[1].status
    np.testing.assert_array_equal(a[0].cpu().numpy(), b[0].cpu().numpy())


def test_cooperative_solve_workspace_without_halo_words():
    f, m = _image(100, 130, seed=1)
    full = fg.workspace_bytes(130, 100)
    out = []
    for nbytes in (full, full - 16 * 100 * 160, full - 16 * 100 * 160 - 256):
        ws = torch.full((nbytes,), 0xA5, dtype=torch.uint8, device=DEV)  # stale contents are ignored
        u = torch.empty_like(f)
        p = fg._params(0.05, 1.0, 0.0, 10, 3)
        st = fg.lib().foeed_inpaint(C.c_void_p(f.data_ptr()), C.c_void_p(m.data_ptr()), C.c_void_p(u.data_ptr()), 130, 100,
                                    130, 0, C.byref(p), C.c_void_p(ws.data_ptr()), nbytes,
                                    C.c_void_p(torch.cuda.current_stream().cuda_stream), None)
        out.append((st, u))
    assert [st for st, _ in out] == [0, 0, 1] and torch.equal(out[0][1], out[1][1])


@pytest.mark.parametrize("method", [0, 1])
# 8 x 4 tiles: one partial tile, edges one pixel wide and high, the smallest side; 8 x 8; 16 x 16 with up to three
# per SM; more than that
@pytest.mark.parametrize("shape", [(16, 16), (17, 25), (64, 64), (16, 1000), (97, 129), (160, 157), (177, 193), (300, 303), (340, 341)])
@pytest.mark.parametrize("sigma", [0.0, 1.0, 2.0])
def test_cooperative_f64_solve_is_the_stepwise_solve(method, shape, sigma):
    f, m = _image(*shape, seed=shape[0])
    _same(*_both(method, f.double(), m, 0.05, sigma, 7, 4))


@pytest.mark.parametrize("kw", [dict(diffusivity=1, mu3_mode=1), dict(diffusivity=2)])
@pytest.mark.parametrize("shape", [(40, 57), (190, 200)])
@pytest.mark.parametrize("n,cycles", [(2, 5), (128, 1), (129, 1)])
def test_cooperative_f64_models_and_cycle_counts(kw, shape, n, cycles):
    f, m = _image(*shape, seed=n)
    _same(*_both(0, f.double(), m, 0.05, 1.5, n, cycles, **kw))


@pytest.mark.parametrize("kw", [dict(tol=1e-3), dict(tau=0.4)])
@pytest.mark.parametrize("shape", [(40, 57), (190, 200)])
def test_cooperative_f64_solve_stops_at_the_same_cycle(kw, shape):
    f, m = _image(*shape, seed=1)
    a, b = _both(0, f.double(), m, 0.05, 1.0, 20, 60, **kw)
    assert a[1].cycles_run == b[1].cycles_run < 60 and a[1].status == b[1].status
    np.testing.assert_array_equal(a[0].cpu().numpy(), b[0].cpu().numpy())


# --------------------------------------------------------------------------
# large images: (step, tile) pairs taken in order in cooperative launches


@pytest.mark.parametrize("method", [0, 1])
# just over four 64 x 32 tiles per SM, ragged; wide and flat; the largest the rule takes; one tile row more
@pytest.mark.parametrize("shape", [(959, 1345), (33, 39050), (1970, 4096), (2017, 4096)])
@pytest.mark.parametrize("sigma", [0.5, 1.5])
def test_flow_solve_is_the_stepwise_solve(method, shape, sigma):
    f, m = _image(*shape, seed=shape[0])
    _same(*_both(method, f, m, 0.05, sigma, 5, 3))


@pytest.mark.parametrize("method", [0, 1])
# 64 x 16 tiles: just over 5.5 per SM, ragged; wide and flat; the largest the rule takes; one tile row more (64 x 32)
@pytest.mark.parametrize("shape", [(419, 1985), (17, 26801), (1008, 1400), (1009, 1400)])
@pytest.mark.parametrize("sigma", [0.5, 2.0])
def test_flow_solve_on_low_tiles(method, shape, sigma):
    f, m = _image(*shape, seed=shape[0])
    _same(*_both(method, f, m, 0.05, sigma, 5, 3))


@pytest.mark.parametrize("shape", [(625, 1000), (630, 1030), (801, 1100)])
@pytest.mark.parametrize("n,cycles", [(2, 4), (7, 3), (100, 22)])
def test_flow_on_low_tiles_with_the_two_float_update(shape, n, cycles):
    f, m = _image(*shape, seed=n)
    _same(*_both(0, f, m, 0.05, 2.0, n, cycles, dtype="f32_f64u"))


@pytest.mark.parametrize("kw", [dict(tol=1e-3), dict(tau=0.4)])
def test_flow_on_low_tiles_stops_at_the_same_cycle(kw):
    f, m = _image(900, 1100, seed=1)
    a, b = _both(0, f, m, 0.05, 1.0, 20, 60, **kw)
    assert a[1].cycles_run == b[1].cycles_run < 60 and a[1].status == b[1].status
    np.testing.assert_array_equal(a[0].cpu().numpy(), b[0].cpu().numpy())


@pytest.mark.parametrize("n,cycles", [(2, 1), (2, 4), (3, 3), (128, 2), (100, 43), (129, 1)])
def test_flow_cycle_counts(n, cycles):
    """Shortest and longest cycles, several launches (100 x 43 steps), one step too many."""
    f, m = _image(1000, 1300, seed=n)
    _same(*_both(0, f, m, 0.05, 1.0, n, cycles))


@pytest.mark.parametrize("kw", [dict(dtype="f32_f64u"), dict(diffusivity=1, mu3_mode=1)])
def test_flow_size_models(kw):
    f, m = _image(1000, 1300, seed=3)
    _same(*_both(0, f, m, 0.05, 2.0, 5, 2, **kw))


@pytest.mark.parametrize("n,tol", [(2, 1e-3), (30, 1e-3)])
def test_flow_solve_stops_at_the_same_cycle(n, tol):
    f, m = _image(1000, 1300, seed=n)
    for method in (0, 1):
        _same(*_both(method, f, m, 0.05, 1.0, n, 60, tol=tol))


def test_flow_solve_stops_where_it_diverges():
    f, m = _image(1000, 1300, seed=1)
    a, b = _both(0, f, m, 0.05, 1.0, 20, 50, tau=0.4)
    assert a[1].status == 4 and a[1].cycles_run == b[1].cycles_run
    np.testing.assert_array_equal(a[0].cpu().numpy(), b[0].cpu().numpy())


def test_flow_solves_beside_other_streams_match_sequential_solves():
    """Two threads with a stream each while a third stream's kernels come and go: CTAs of a cooperative launch may
    start after others have ended cycles."""
    cases = [(0, 6, 50, {}), (1, 7, 50, dict(tol=1e-4)), (0, 6, 40, dict(dtype="f32_f64u"))]
    images = [_image(1000, 1300, seed=5), _image(840, 1100, seed=6)]

    def solve(f, m, case, **kw):
        method, n, cycles, opt = case
        fn = fg.foeed_inpaint if method == 0 else fg.eed_inpaint
        return fn(f, m, 0.05, 1.0, n, cycles, raise_on_status=False, **opt, **kw)

    ref = [[solve(f, m, c) for c in cases] for f, m in images]
    torch.cuda.synchronize(DEV)
    got, routes, errors = {}, [], []

    def worker(i):
        try:
            s = torch.cuda.Stream(device=DEV)
            for rep in range(3):
                for j, c in enumerate(cases):
                    got[i, rep, j] = solve(*images[i], c, stream=s)
                    routes.append(fg.last_route())
            s.synchronize()
        except Exception as e:  # reported below
            errors.append(e)

    other = torch.cuda.Stream(device=DEV)
    buf = torch.ones(1 << 26, device=DEV)
    other.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(other):
        for _ in range(400):  # some 40 ms of kernels that fill the GPU
            buf.mul_(1.0)
    ts = [threading.Thread(target=worker, args=(i,)) for i in range(2)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    torch.cuda.synchronize(DEV)
    assert not errors, errors
    assert len(got) == 2 * 3 * len(cases)
    assert all(r["kind"] == "ordered" and not r["gave_up"] for r in routes), routes
    for (i, rep, j), a in got.items():
        _same(a, ref[i][j])


# --------------------------------------------------------------------------
# the route of a solve, and a cooperative launch that gives up

# method, keywords, shape, kind and tile
ROUTES = [(0, {}, (250, 511), "resident", (64, 8)), (1, {}, (512, 515), "resident", (64, 16)),
          (0, dict(dtype="f32_f64u"), (700, 701), "resident", (64, 16)), (0, {}, (720, 1280), "resident", (64, 24)),
          (0, dict(diffusivity=1, mu3_mode=1), (300, 400), "resident", (64, 8)),
          (0, dict(dtype="f64"), (64, 64), "resident", (8, 4)), (1, dict(dtype="f64"), (200, 200), "resident", (16, 16)),
          (0, {}, (1000, 1300), "ordered", (64, 16)), (1, {}, (1080, 1920), "ordered", (64, 32)),
          (0, dict(diffusivity=1), (1000, 1300), "steps", None), (0, dict(dtype="f64"), (512, 512), "steps", None),
          (0, {}, (3000, 2900), "steps", None)]


@pytest.mark.parametrize("method,kw,shape,kind,tile", ROUTES)
def test_route_of_a_solve_and_of_one_that_gives_up(method, kw, shape, kind, tile):
    """A wait limit of one poll: the kernel leaves with its status, and the solve is repeated step by step from its
    inputs, u0 among them, with the same bits. Without cooperative launches the limit changes nothing."""
    f, m = _image(*shape, seed=8)
    kw = dict(kw, u0=torch.flip(f, (0,)))
    a, b = _both(method, f, m, 0.05, 1.0, 12, 5, **kw)
    solve = fg.foeed_inpaint if method == 0 else fg.eed_inpaint
    again = solve(f, m, 0.05, 1.0, 12, 5, **kw)
    route = fg.last_route()
    assert (route["kind"], route["gave_up"]) == (kind, False)
    assert tile is None or (route["tile_w"], route["tile_h"]) == tile
    fg.set_wait_limit(1)
    try:
        c = solve(f, m, 0.05, 1.0, 12, 5, **kw)
        route = fg.last_route()
    finally:
        fg.set_wait_limit(0)
    assert (route["kind"], route["gave_up"]) == ("steps", kind != "steps")
    for x in (a, again, c):
        _same(x, b)


def _kind(method, shape, sigma, n, cycles, **kw):
    f, m = _image(*shape, seed=1)
    (fg.foeed_inpaint if method == 0 else fg.eed_inpaint)(f, m, 0.05, sigma, n, cycles, raise_on_status=False, **kw)
    return fg.last_route()["kind"]


@pytest.mark.parametrize("method", [0, 1])
@pytest.mark.parametrize("dtype,more", [("f32", "steps"), ("f32_f64u", "ordered")])
def test_wide_gaussian_on_24_high_tiles_to_three_per_sm(method, dtype, more):
    """456 tiles of 64 x 24 and 460, the same for both methods."""
    assert _kind(method, (576, 1216), 2.0, 12, 2, dtype=dtype) == "resident"
    assert _kind(method, (552, 1280), 2.0, 12, 2, dtype=dtype) == more


# n, cycles, route: few steps in a launch and short cycles are left to the step kernels
@pytest.mark.parametrize("shape,n,cycles,kind", [
    ((700, 701), 3, 1, "steps"), ((700, 701), 2, 2, "resident"), ((300, 400), 2, 1, "resident"),
    ((1000, 1300), 5, 20, "steps"), ((1000, 1300), 9, 1, "steps"), ((1000, 1300), 6, 2, "ordered"),
    ((1080, 1920), 3, 20, "steps"), ((1080, 1920), 4, 1, "steps"), ((1080, 1920), 4, 2, "ordered")])
def test_route_by_the_number_of_steps(shape, n, cycles, kind):
    f, m = _image(*shape, seed=n)
    a, b = _both(0, f, m, 0.05, 1.0, n, cycles)
    _same(a, b)
    assert _kind(0, shape, 1.0, n, cycles) == kind


@pytest.mark.parametrize("shape,n,kind", [((700, 701), 3, "steps"), ((700, 701), 4, "resident"), ((1000, 1300), 9, "steps"),
                                          ((1000, 1300), 10, "ordered"), ((1080, 1920), 7, "steps"), ((1080, 1920), 8, "ordered")])
def test_route_of_kept_states_by_the_cycle_length(shape, n, kind):
    f, m = _image(*shape, seed=n)
    x = f.clone().requires_grad_(True)
    u = fg.foeed_inpaint_diff(x, m, 0.05, 1.0, n, 4)
    assert fg.last_route()["kind"] == kind
    (g,) = torch.autograd.grad(u, x, torch.ones_like(u))
    ref, uref = fg.foeed_inpaint_vjp(f, m, torch.ones_like(f), 0.05, 1.0, n, 4)
    assert torch.equal(u.detach(), uref) and torch.equal(g, ref)


@pytest.mark.parametrize("method,kw,sigma,shape,kind", [
    (0, {}, 1.5, (2176, 3200), "ordered"), (0, {}, 1.5, (2177, 3200), "steps"), (0, {}, 2.0, (2177, 3200), "ordered"),
    (1, {}, 1.5, (2177, 3200), "ordered"), (0, dict(dtype="f32_f64u"), 1.0, (2177, 3200), "ordered")])
def test_largest_ordered_solves(method, kw, sigma, shape, kind):
    """3400 tiles of 64 x 32 and one row of tiles more."""
    f, m = _image(*shape, seed=3)
    _same(*_both(method, f, m, 0.05, sigma, 4, 2, **kw))
    assert _kind(method, shape, sigma, 4, 2, **kw) == kind


@pytest.mark.parametrize("method", [0, 1])
# the edges of the ordered kernel's tiles (64 x 16, then 64 x 32) in cycles that it takes
@pytest.mark.parametrize("shape", [(801, 1217), (33, 26801), (1008, 1400), (1009, 1400), (959, 1345), (33, 39050)])
@pytest.mark.parametrize("sigma", [0.5, 2.0])
def test_ordered_solve_at_tile_edges(method, shape, sigma):
    f, m = _image(*shape, seed=shape[0])
    _same(*_both(method, f, m, 0.05, sigma, 6, 3))
    assert _kind(method, shape, sigma, 6, 3) == "ordered"


# sizes and cycles that run step by step: the autotuner and the graph cache

@pytest.mark.parametrize("method,kw", [(0, {}), (1, {}), (0, dict(diffusivity=1, mu3_mode=1))])
# under one 64 x 32 tile per SM; one to four (the later triggers too); wide and flat; more than four
@pytest.mark.parametrize("shape", [(300, 515), (625, 1031), (97, 2111), (1201, 1999)])
def test_autotuner_on_stepwise_solves(method, kw, shape):
    """Cycles of one step are timed: the plan says so, the choice is the fastest and is kept, and every tile shape gives
    the same bits."""
    f, m = _image(*shape, seed=6)
    solve = fg.foeed_inpaint if method == 0 else fg.eed_inpaint
    two = method == 1 or bool(kw)  # 64 x 32 and 64 x 16 tiles only
    ua, _ = solve(f, m, 0.05, 1.5, 1, 12, **kw)
    plan = fg.last_tile_plan()
    assert fg.last_route()["kind"] == "steps" and plan["tuned"] == 1
    times = {32: plan["us_h32"], 16: plan["us_h16"]}
    if not two:
        times.update({64: plan["us_h64"], 8: plan["us_h8"]})
    assert all(t > 0 for t in times.values())
    assert plan["us_chosen"] == min(times.values()) == times[plan["tile_h"]]
    ub, _ = solve(f, m, 0.05, 1.5, 1, 12, **kw)
    again = fg.last_tile_plan()
    assert again["tuned"] == 0 and again["tile_h"] == plan["tile_h"] and torch.equal(ua, ub)
    try:
        for pol, th in (("h32", 32), ("h16", 16), ("h64", 32 if two else 64), ("h8", 16 if two else 8)):
            fg.set_tile_policy(pol)
            u, _ = solve(f, m, 0.05, 1.5, 1, 12, **kw)
            assert fg.last_tile_plan()["tile_h"] == th and torch.equal(u, ua), pol
    finally:
        fg.set_tile_policy("auto")


def test_graph_caches_of_two_threads_evict():
    """Six graph keys per thread, cycles of 130 steps: more than the four entries of a thread's cache."""
    f, m = _image(64, 96, seed=3)
    lams = [0.02 * (i + 1) for i in range(6)]
    ref = {lam: fg.foeed_inpaint(f, m, lam, 1.0, 130, 2)[0].clone() for lam in lams}
    got, kinds, errors = {}, [], []

    def worker(tid):
        try:
            s = torch.cuda.Stream(device=DEV)
            for rep in range(2):
                for lam in (lams if tid == 0 else lams[::-1]):
                    got[tid, rep, lam] = fg.foeed_inpaint(f, m, lam, 1.0, 130, 2, stream=s)[0]
                    kinds.append(fg.last_route()["kind"])
            s.synchronize()
        except Exception as e:  # reported below
            errors.append(e)

    torch.cuda.synchronize(DEV)
    ts = [threading.Thread(target=worker, args=(t,)) for t in range(2)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not errors, errors
    assert len(got) == 24 and set(kinds) == {"steps"}
    for (tid, rep, lam), u in got.items():
        assert torch.equal(u, ref[lam]), (tid, rep, lam)


def test_differentiable_solve_that_gives_up():
    f, m = _image(300, 400, seed=9)
    grads = []
    for polls in (0, 1):
        x = f.clone().requires_grad_(True)
        fg.set_wait_limit(polls)
        try:
            u = fg.foeed_inpaint_diff(x, m, 0.05, 1.0, 10, 4)
            assert fg.last_route()["gave_up"] == (polls == 1)
        finally:
            fg.set_wait_limit(0)
        grads.append((u.detach(), torch.autograd.grad(u, x, torch.cos(7.0 * u.detach()))[0]))
    assert torch.equal(grads[0][0], grads[1][0]) and torch.equal(grads[0][1], grads[1][1])


# --------------------------------------------------------------------------
# gradient from the iterates kept at the start of every cycle


@pytest.mark.parametrize("shape", [(16, 16), (5, 9), (70, 131), (520, 600)])
@pytest.mark.parametrize("n,cycles,keep", [(1, 6, True), (7, 5, True), (40, 2, True), (300, 1, False)])
@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
def test_gradient_from_kept_states_is_the_vjp(shape, n, cycles, keep, dtype):
    """Against the gradient that runs its own forward solve; pitched rows; two backward passes. 300 steps in one
    cycle would hold more images than the checkpoints: the forward keeps nothing."""
    if dtype == torch.float64 and shape[0] > 100:
        pytest.skip("the FP32 shape")
    h, w = shape
    f, m = _image(h, w, seed=n)
    f = torch.empty_strided((h, w), (w + 5, 1), dtype=dtype, device=DEV).copy_(f).requires_grad_(True)
    assert fg._keeps_states(f, m, n, cycles, 16) == keep
    u = fg.foeed_inpaint_diff(f, m, 0.05, 1.0, n, cycles)
    gu = torch.cos(7.0 * u.detach())
    (g1,) = torch.autograd.grad(u, f, gu, retain_graph=True)
    (g2,) = torch.autograd.grad(u, f, gu)
    ref, uref = fg.foeed_inpaint_vjp(f.detach(), m, gu, 0.05, 1.0, n, cycles)
    assert torch.equal(u.detach(), uref) and torch.equal(g1, ref) and torch.equal(g2, ref)


@pytest.mark.parametrize("mode", [torch.no_grad, torch.inference_mode, torch.enable_grad])
def test_iterates_are_kept_only_where_a_gradient_is_recorded(mode, monkeypatch):
    calls, states_call = [], fg._states_call
    monkeypatch.setattr(fg, "_states_call", lambda *a: (calls.append(a[0]), states_call(*a)))
    f, m = _image(70, 131, seed=2)
    ref, _ = fg.foeed_inpaint(f, m, 0.05, 1.0, 10, 4)
    x = f.clone().requires_grad_(True)
    with mode():
        u = fg.foeed_inpaint_diff(x, m, 0.05, 1.0, 10, 4)
    assert torch.equal(u.detach(), ref) and calls == (["solve"] if mode is torch.enable_grad else [])


def test_kept_states_argument_errors():
    f, m = _image(20, 30, seed=1)
    L, p = fg.lib(), fg._params(0.05, 1.0, 0.0, 4, 3)
    n = int(L.foeed_states_bytes(30, 20, 0, C.byref(p)))
    assert n == 3 * 20 * 32 * 4 and L.foeed_states_bytes(30, 20, 2, C.byref(p)) == 0
    ws = torch.empty(fg.workspace_bytes(30, 20), dtype=torch.uint8, device=DEV)
    states, u = torch.empty(n, dtype=torch.uint8, device=DEV), torch.empty_like(f)

    def call(nbytes, prm, dtype=0):
        return L.foeed_inpaint_states(C.c_void_p(f.data_ptr()), C.c_void_p(m.data_ptr()), C.c_void_p(u.data_ptr()), 30, 20,
                                      30, dtype, C.byref(prm), C.c_void_p(states.data_ptr()), nbytes,
                                      C.c_void_p(ws.data_ptr()), ws.numel(),
                                      C.c_void_p(torch.cuda.current_stream().cuda_stream), None)

    assert call(n, p) == 0
    assert call(n - 1, p) == 1
    assert call(n, fg._params(0.05, 1.0, 0.0, 4, 3, tol=1e-3)) == 1
    assert call(n, p, dtype=2) == 1
    assert call(n, fg._params(0.05, 1.0, 0.5, 40, 3)) in (0, 4)  # a diverging solve is reported, as by foeed_inpaint
