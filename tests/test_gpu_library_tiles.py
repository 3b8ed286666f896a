"""GPU: the tiles the library chooses by itself, at the sizes where they can go
wrong: the tensor-core collision filter (reg = 0), the row tiles of the FP32
distance map (reg = 0), Life runs of more than 16 steps, the fused cost-model
kernels and the scaled FP16 planes of the tensor-core distance map."""
import numpy as np
import pytest

from gpu_util import dev, rel_err, tri
from paper_1609_01490_gb300 import inputs

pytestmark = pytest.mark.gpu


# --------------------------------------------------------------- collisions --
def _collide(c, r, map_id, cap):
    import torch
    t, D, n = tri(), dev(), c.shape[0]
    npairs = torch.full((1,), 9, dtype=torch.int64, device=D)
    count = torch.full((n,), 7, dtype=torch.int32, device=D)
    pairs = torch.zeros((cap, 2), dtype=torch.int32, device=D) if cap else None
    t.tri_collide(torch.from_numpy(np.ascontiguousarray(c)).to(D), torch.from_numpy(np.ascontiguousarray(r)).to(D),
                  npairs, count=count, pairs=pairs, map=map_id)
    torch.cuda.synchronize()
    pl = pairs[:int(npairs.item())].cpu().numpy().astype(np.int64) if cap else None
    return int(npairs.item()), count.cpu().numpy().astype(np.uint32), pl


def _check_collide(orc, c, r, maps=("LAMBDA",)):
    cnt_ref, pi, pj = orc.collide_counts(c, r)
    n = c.shape[0]
    for name in maps:
        for cap in (0, len(pi) + 1):
            tot, cnt, pl = _collide(c, r, getattr(tri(), "MAP_" + name), cap)
            assert tot == len(pi), (name, cap)
            np.testing.assert_array_equal(cnt, cnt_ref)
            if cap:
                np.testing.assert_array_equal(np.sort(pl[:, 0] * n + pl[:, 1]), np.sort(pi * n + pj))


@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("n", [1, 2, 63, 64, 65, 127, 128, 129, 257, 1000])
def test_collide_filter_tile_edges(orc, dim, n):
    c, r = inputs.spheres(n, dim, kappa=8.0, seed=n + dim)
    _check_collide(orc, c, r, ("LAMBDA", "LAMBDA_PDELTA", "BB", "RB", "REC") if n <= 128 else ("LAMBDA", "BB"))


@pytest.mark.parametrize("n", [6400, 18000])  # 256- and 512-sphere tiles
def test_collide_filter_larger_tiles(orc, n):
    c, r = inputs.spheres(n, 3, kappa=4.0, seed=n)
    _check_collide(orc, c, r, ("LAMBDA", "RB"))


@pytest.mark.parametrize("case", ["offset", "tiny", "huge", "overflow", "crowd", "special", "point"])
def test_collide_filter_scales(orc, case):
    # far from the origin, extents at and past the filter's range, most spheres in a
    # small part of the extent (which gives the filter up), infinities and NaNs
    c, r = inputs.spheres(700, 3, kappa=10.0, seed=11)
    if case == "offset":
        c = (c + np.float32(3000.0)).astype(np.float32)
    elif case == "tiny":
        c, r = (c * np.float32(2.0 ** -70)).astype(np.float32), (r * np.float32(2.0 ** -70)).astype(np.float32)
    elif case == "huge":
        c, r = (c * np.float32(2.0 ** 59)).astype(np.float32), (r * np.float32(2.0 ** 59)).astype(np.float32)
    elif case == "overflow":
        c, r = (c * np.float32(2.0 ** 100)).astype(np.float32), (r * np.float32(2.0 ** 100)).astype(np.float32)
    elif case == "crowd":
        c = c.copy()
        c[::97] *= np.float32(4000.0)
    elif case == "special":
        c, r = c.copy(), r.copy()
        c[5, 1], c[140, 0], r[33], r[300] = np.inf, np.nan, np.inf, np.nan
    else:
        c = np.full_like(c, 0.25)
    with np.errstate(all="ignore"):
        _check_collide(orc, c, r)


@pytest.mark.parametrize("dim", [1, 2, 3])
@pytest.mark.parametrize("reg", [0, 4, 8])
def test_collide_exact_touch(orc, dim, reg):
    """Pairs that touch exactly, s = q after rounding: their squares round up and
    down alike.  Packed products fused into the next sum would miss half of them."""
    import torch
    t, D, n = tri(), dev(), 1400
    rng = np.random.default_rng(dim)
    gap = rng.integers(1 << 12, 1 << 14, n // 2) * 2.0 ** -12  # 13-bit gaps: differences and sums are exact
    c = np.zeros((n, dim))
    c[::2, 0] = 5.0 * np.arange(n // 2)
    c[1::2, 0] = c[::2, 0] + gap
    r = np.repeat(gap / 2, 2)
    order = np.concatenate([np.arange(0, n, 2), np.arange(1, n, 2)])  # partners far apart, no diagonal pair beside them
    c, r = c[order], r[order]
    scale = np.float32(1.1)  # 24-bit values, each pair still at equal rounded distance and radius sum or apart
    for c32, r32 in ((c.astype(np.float32), r.astype(np.float32)),
                     ((c * (2 ** 12 + 1)).astype(np.float32) * scale, (r * (2 ** 12 + 1)).astype(np.float32) * scale)):
        cnt_ref, pi, _ = orc.collide_counts(c32, r32)
        npairs = torch.zeros(1, dtype=torch.int64, device=D)
        count = torch.zeros(n, dtype=torch.int32, device=D)
        t.tri_collide(torch.from_numpy(c32).to(D), torch.from_numpy(r32).to(D), npairs, count=count, reg=reg)
        assert npairs.item() == len(pi)
        np.testing.assert_array_equal(count.cpu().numpy().astype(np.uint32), cnt_ref)


@pytest.mark.parametrize("reg", [4, 8])
@pytest.mark.parametrize("e", [-70, -66, 0, 61, 80])
def test_collide_packed_tile_scales(orc, reg, e):
    # squares that vanish or overflow in FP32, and radii of either sign, through the
    # packed tile itself
    import torch
    t, D, n = tri(), dev(), 500
    for dim in (2, 3):
        c, r = inputs.spheres(n, dim, kappa=4.0, seed=n + dim)
        c, r = np.ldexp(c, e).astype(np.float32), np.ldexp(r, e).astype(np.float32)
        if e == 0:
            r[::3] *= np.float32(-0.75)
        r[7] = np.inf
        with np.errstate(all="ignore"):
            cnt_ref, pi, _ = orc.collide_counts(c, r)
        npairs = torch.zeros(1, dtype=torch.int64, device=D)
        count = torch.zeros(n, dtype=torch.int32, device=D)
        t.tri_collide(torch.from_numpy(c).to(D), torch.from_numpy(r).to(D), npairs, count=count, reg=reg)
        assert npairs.item() == len(pi)
        np.testing.assert_array_equal(count.cpu().numpy().astype(np.uint32), cnt_ref)


@pytest.mark.parametrize("n", [6401, 18001])  # 256- and 512-sphere tiles, ragged ends
@pytest.mark.parametrize("case", ["crowd", "tiny", "special"])
def test_collide_filter_gives_up_at_larger_tiles(orc, n, case):
    # the packed FP32 tiles inside a larger block: the skips above the diagonal and past n
    c, r = inputs.spheres(n, 3, kappa=4.0, seed=n)
    c, r = c.copy(), r.copy()
    if case == "crowd":
        c[::97] *= np.float32(4000.0)
    elif case == "tiny":
        c, r = np.ldexp(c, -70).astype(np.float32), np.ldexp(r, -70).astype(np.float32)
    else:
        c[::3, 1] = np.nan
        c[5, 0], r[33], r[n - 1] = np.inf, np.inf, np.nan
    with np.errstate(all="ignore"):
        _check_collide(orc, c, r, ("LAMBDA", "RB"))


# ------------------------------------------------------------ FP32 distances --
@pytest.mark.parametrize("d", [1, 2, 3, 4, 5, 8])
@pytest.mark.parametrize("n", [1, 3, 125, 126, 127, 128, 129, 256, 383, 700])
def test_edm_row_tiles(d, n):
    # the same operations per pair as the 4 x 4 tile: the same bits, at every
    # alignment of the output, and nothing written around it
    import torch
    t, D = tri(), dev()
    x = torch.from_numpy(inputs.edm_normal_points(n, d, seed=n + d)).to(D)
    size = n * (n + 1) // 2
    ref = torch.empty(size, device=D)
    t.tri_edm(x, ref, reg=4)
    for name in ("LAMBDA", "LAMBDA_PDELTA", "BB", "RB"):
        for off in range(4):
            buf = torch.full((size + 16,), -7.0, device=D)
            t.tri_edm(x, buf[8 + off:8 + off + size], map=getattr(t, "MAP_" + name))
            assert torch.equal(buf[8 + off:8 + off + size], ref), (name, off)
            assert bool((buf[:8 + off] == -7.0).all()) and bool((buf[8 + off + size:] == -7.0).all())


@pytest.mark.parametrize("d", [1, 2, 3, 4, 5, 8])
@pytest.mark.parametrize("n", [6145, 6271, 6272])  # one, 127 and 128 rows in the last tile row
def test_edm_row_tiles_at_chosen_sizes(d, n):
    # sizes at which tri_edm takes the row tile by itself, for every d <= 8
    import torch
    t, D = tri(), dev()
    x = torch.from_numpy(inputs.edm_normal_points(n, d, seed=n + d)).to(D)
    size = n * (n + 1) // 2
    ref = torch.empty(size, device=D)
    t.tri_edm(x, ref, reg=4)
    for name in ("LAMBDA", "RB"):
        for off in range(4):
            buf = torch.full((size + 16,), -7.0, device=D)
            t.tri_edm(x, buf[8 + off:8 + off + size], map=getattr(t, "MAP_" + name))
            assert torch.equal(buf[8 + off:8 + off + size], ref), (name, off)
            assert bool((buf[:8 + off] == -7.0).all()) and bool((buf[8 + off + size:] == -7.0).all())


@pytest.mark.parametrize("d,sizes", [(1, (4993, 5119, 5120)), (2, (4993,)), (3, (4993, 5119, 5120)), (4, (5121,)),
                                     (5, (6145,)), (6, (6271,)), (7, (6272,)), (8, (6145, 6273))])
def test_edm_row_tiles_under_every_map(d, sizes):
    # the smallest sizes that take the row tile, one row more or less in its last tile row
    import torch
    t, D = tri(), dev()
    for n in sizes:
        x = torch.from_numpy(inputs.edm_normal_points(n, d, seed=n + d)).to(D)
        size = n * (n + 1) // 2
        ref = torch.empty(size, device=D)
        t.tri_edm(x, ref, reg=4)
        for k, name in enumerate(("LAMBDA", "LAMBDA_PDELTA", "BB", "RB")):
            off = (n + k) % 4
            buf = torch.full((size + 16,), -7.0, device=D)
            t.tri_edm(x, buf[8 + off:8 + off + size], map=getattr(t, "MAP_" + name))
            assert torch.equal(buf[8 + off:8 + off + size], ref), (n, name)
            assert bool((buf[:8 + off] == -7.0).all()) and bool((buf[8 + off + size:] == -7.0).all())


@pytest.mark.parametrize("d", [9, 16, 33, 100])
def test_edm_chosen_square_tiles(d):
    # sizes on both sides of the choice between 4 x 4 and 8 x 8 pairs per thread
    import torch
    t, D = tri(), dev()
    for n in (300, 5000):
        x = torch.from_numpy(inputs.edm_normal_points(n, d, seed=n + d)).to(D)
        a, b = (torch.empty(n * (n + 1) // 2, device=D) for _ in range(2))
        for rho in (8, 16, 32):
            t.tri_edm(x, a, rho=rho)
            t.tri_edm(x, b, rho=rho, reg=4)
            assert torch.equal(a, b), (n, rho)


@pytest.mark.parametrize("prec", ["BF16X6", "BF16X3"])
def test_tc_edm_row_scales(orc, prec):
    # rows from 2^-40 to 2^40, zero rows, rows whose largest feature dwarfs the
    # others: every distance within the 1e-5 the split is built for
    import torch
    t, D = tri(), dev()
    n, d = 400, 96
    x = inputs.edm_normal_points(n, d, seed=5)
    rng = np.random.default_rng(7)
    x = (x * np.exp2(rng.integers(-40, 41, size=(n, 1)))).astype(np.float32)
    x[::37] = 0.0
    x[3::29, 0] *= np.float32(2.0 ** 20)
    out = torch.empty(n * (n + 1) // 2, device=D)
    p = getattr(t, prec)
    ws = torch.empty(t.tri_edm_workspace_size(n, d, p), dtype=torch.uint8, device=D)
    t.tri_edm(torch.from_numpy(x).to(D), out, prec=p, workspace=ws)
    assert rel_err(out.cpu().numpy(), orc.edm_packed(x)) <= 1e-5


# --------------------------------------------------------------------- Life --
@pytest.mark.parametrize("mapname", ["LAMBDA", "LAMBDA_PDELTA", "BB", "RB", "REC"])
@pytest.mark.parametrize("n", [60, 95, 112, 113, 192, 224, 240, 337, 448, 1000])
def test_life_long_runs_at_tile_edges(orc, mapname, n):
    # 96- and 112-cell tiles: sizes around them, more than 16 steps, cells of any
    # non-zero byte, junk outside the domain that must come back unchanged
    import torch
    t, D = tri(), dev()
    m = -(-n // 128)
    if mapname == "REC" and m & (m - 1):
        pytest.skip("REC needs a power of two of 128-cell block rows")
    ld = -(-n // 16) * 16 + 16
    g = inputs.ca_grid(n, seed=n, ld=ld)
    g[g != 0] = np.arange(1, 256, dtype=np.uint8)[np.arange(int((g != 0).sum())) % 255]
    g[np.triu_indices(n, 1)] = 5
    g[:, n:] = 9
    a = torch.from_numpy(g).to(D)
    for steps in (17, 24, 33, 50):
        out, scratch = a.clone(), torch.full_like(a, 7)
        t.tri_ca_run(a, out, n, steps, scratch=scratch, map=getattr(t, "MAP_" + mapname))
        assert np.array_equal(out.cpu().numpy(), orc.ca_run(g, steps)), steps
        s = scratch.cpu().numpy()
        assert np.all(s[np.triu_indices(n, 1)] == 7) and np.all(s[:, n:] == 7)


@pytest.mark.parametrize("n", [5999, 6001, 9000])
def test_life_long_runs_match_single_steps(n):
    # both halos at sizes with many tiles, against step-by-step tri_ca_step
    import torch
    t, D = tri(), dev()
    ld = -(-n // 16) * 16
    a = torch.randint(0, 2, (n, ld), generator=torch.Generator(device=D).manual_seed(n), device=D, dtype=torch.uint8).tril_()
    out, scratch, p, q = (torch.zeros_like(a) for _ in range(4))
    t.tri_ca_run(a, out, n, 35, scratch=scratch)
    src = a
    for s in range(35):
        dst = q if s & 1 else p
        t.tri_ca_step(src, dst, n, rho=32)
        src = dst
    assert torch.equal(out, src)


@pytest.mark.parametrize("n", [1, 63, 64, 65, 128, 129, 1000, 3001])
@pytest.mark.parametrize("rho", [8, 16, 32])
def test_life_step_default_tiles(orc, n, rho):
    import torch
    t, D = tri(), dev()
    ld = -(-n // 16) * 16
    g = inputs.ca_grid(n, seed=n, ld=ld)
    g[np.triu_indices(n, 1)] = 5
    a = torch.from_numpy(g).to(D)
    ref = orc.ca_step(g)
    for name in ("LAMBDA", "BB", "RB"):
        out = a.clone()
        t.tri_ca_step(a, out, n, map=getattr(t, "MAP_" + name), rho=rho)
        assert np.array_equal(out.cpu().numpy(), ref), name


@pytest.mark.parametrize("n", [1, 65, 1000, 5999, 6000, 6001])
@pytest.mark.parametrize("rule", ["life", "highlife"])
def test_life_step_tiles_agree(orc, n, rule):
    # both sides of the size from which Conway's rule takes one tile whatever rho, and
    # every tile asked for by itself
    import torch
    t, D = tri(), dev()
    birth, survive = (t.LIFE_BIRTH, t.LIFE_SURVIVE) if rule == "life" else ((1 << 3) | (1 << 6), (1 << 2) | (1 << 3))
    ld = -(-n // 16) * 16
    g = inputs.ca_grid(n, seed=n, ld=ld)
    if n <= 1000:
        g[np.triu_indices(n, 1)] = 5
    a = torch.from_numpy(g).to(D)
    ref = torch.from_numpy(orc.ca_step(g, birth, survive)).to(D)
    for rho in (8, 16, 32):
        for name in ("LAMBDA", "LAMBDA_PDELTA", "BB", "RB"):
            for call in (t.tri_ca_step, t.tri_ca_step_tile):
                out = a.clone()
                call(a, out, n, birth_mask=birth, survive_mask=survive, map=getattr(t, "MAP_" + name), rho=rho)
                assert torch.equal(out, ref), (rho, name, call.__name__)


# ------------------------------------------------------------- host threads --
def test_calls_of_different_sizes_from_threads():
    """Kernels that take more shared memory than by default, at sizes that differ from
    thread to thread: no call lowers the limit under another's launch."""
    import threading

    import torch
    t, D = tri(), dev()
    errors = []

    def forward(F, h1, h2):
        theta = torch.zeros(h1 * F + h1 + h2 * h1 + 2 * h2 + 1, device=D)
        X, pred = torch.zeros(8, F, device=D), torch.zeros(8, device=D)
        ws = torch.empty(t.tri_mlp_workspace_size(8, h1, h2) // 4, device=D)
        for _ in range(20000):
            t.tri_mlp_forward(theta, X, pred, h1, h2, ws)

    def distances(d, prec):
        x, out = torch.randn(200, d, device=D), torch.empty(200 * 201 // 2, device=D)
        ws = torch.empty(t.tri_edm_workspace_size(200, d, prec), dtype=torch.uint8, device=D)
        for _ in range(4000):
            t.tri_edm(x, out, prec=prec, workspace=ws)

    def run(f, *args):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                f(*args)
        except t.TriError as e:
            errors.append(str(e))

    jobs = [(forward, 64, 128, 128), (forward, 14, 128, 96), (forward, 14, 128, 96), (distances, 64, t.BF16X6),
            (distances, 320, t.BF16X3)]
    threads = [threading.Thread(target=run, args=j) for j in jobs]
    for th in threads:
        th.start()
    for th in threads:
        th.join()
    torch.cuda.synchronize()
    assert not errors


# --------------------------------------------------------------- cost model --
@pytest.mark.parametrize("B,F,H1,H2", [(1, 1, 1, 1), (3, 14, 16, 17), (5, 64, 128, 128), (128, 15, 16, 31), (129, 14, 64, 64),
                                       (1030, 14, 33, 96)])
def test_mlp_shapes(orc, B, F, H1, H2):
    import torch
    t, D = tri(), dev()
    rng = np.random.default_rng(B + F)
    theta = (rng.normal(size=orc.mlp_nparams(F, H1, H2)) * 0.2).astype(np.float32)
    X, y = rng.normal(size=(B, F)).astype(np.float32), rng.normal(size=B).astype(np.float32)
    th, Xd, yd = (torch.from_numpy(a).to(D) for a in (theta, X, y))
    ws = torch.empty(t.tri_mlp_workspace_size(B, H1, H2) // 4, device=D)
    pred, loss, grad = torch.empty(B, device=D), torch.empty(1, device=D), torch.full_like(th, 9.0)
    t.tri_mlp_forward(th, Xd, pred, H1, H2, ws)
    t.tri_mlp_grad(th, Xd, yd, loss, grad, H1, H2, ws)
    # sums of at most 129 products and of B terms in FP32: 1e-4 of the scale, as for the fixed shape
    np.testing.assert_allclose(pred.cpu().numpy(), orc.mlp_forward(theta.astype(np.float64), X, H1, H2), rtol=1e-4, atol=1e-5)
    ref_loss, ref_g = orc.mlp_grad(theta.astype(np.float64), X, y, H1, H2)
    assert float(loss.item()) == pytest.approx(ref_loss, rel=1e-5)
    assert np.max(np.abs(grad.cpu().numpy().astype(np.float64) - ref_g)) <= 1e-4 * np.max(np.abs(ref_g))


@pytest.mark.parametrize("B", [4096, 4097, 9001, 40000])
@pytest.mark.parametrize("F,H1,H2", [(3, 8, 5), (14, 32, 17), (14, 64, 64)])
def test_mlp_large_batches(orc, B, F, H1, H2):
    # from 4097 samples on narrow layers take more of them to a block, up to 32
    import torch
    t, D = tri(), dev()
    rng = np.random.default_rng(B + F)
    theta = (rng.normal(size=orc.mlp_nparams(F, H1, H2)) * 0.2).astype(np.float32)
    X, y = rng.normal(size=(B, F)).astype(np.float32), rng.normal(size=B).astype(np.float32)
    th, Xd, yd = (torch.from_numpy(a).to(D) for a in (theta, X, y))
    ws = torch.empty(t.tri_mlp_workspace_size(B, H1, H2) // 4, device=D)
    pred, loss, grad = torch.full((B,), 9.0, device=D), torch.empty(1, device=D), torch.full_like(th, 9.0)
    t.tri_mlp_forward(th, Xd, pred, H1, H2, ws)
    t.tri_mlp_grad(th, Xd, yd, loss, grad, H1, H2, ws)
    # as in test_mlp_shapes
    np.testing.assert_allclose(pred.cpu().numpy(), orc.mlp_forward(theta.astype(np.float64), X, H1, H2), rtol=1e-4, atol=1e-5)
    ref_loss, ref_g = orc.mlp_grad(theta.astype(np.float64), X, y, H1, H2)
    assert float(loss.item()) == pytest.approx(ref_loss, rel=1e-5)
    assert np.max(np.abs(grad.cpu().numpy().astype(np.float64) - ref_g)) <= 1e-4 * np.max(np.abs(ref_g))


@pytest.mark.parametrize("e", [-45, -27, 0, 56])  # sums of squares below 2^-60, about it, ordinary, above 2^100
@pytest.mark.parametrize("d", [1, 3, 32, 33, 100])
def test_tc_edm_recomputed_pairs(d, e):
    """Close and equal pairs are recomputed to within the final rounding (half an
    ulp; the sum's own error is below 2^-40) at every scale."""
    import torch
    t, D = tri(), dev()
    n, rng = 300, np.random.default_rng(d)
    a = rng.normal(size=(n // 2, d)) + np.where(rng.random((n // 2, d)) < 0.5, -3.0, 3.0)
    x = np.stack([a, a + 0.1 * rng.normal(size=a.shape)], 1).reshape(n, d).astype(np.float32)
    x[1:60:2] = x[0:60:2]
    x = np.ldexp(x, e).astype(np.float32)
    xd = torch.from_numpy(x).to(D)
    out = torch.empty(n * (n + 1) // 2, device=D)
    flagged = torch.zeros(1, dtype=torch.int64, device=D)
    ws = torch.empty(t.tri_edm_workspace_size(n, d, t.BF16X3), dtype=torch.uint8, device=D)
    t.tri_edm(xd, out, prec=t.BF16X3, workspace=ws, n_flagged=flagged)
    i = np.arange(1, n, 2)
    got = out.cpu().numpy()[i * (i + 1) // 2 + i - 1]
    want = np.sqrt(((x[i].astype(np.float64) - x[i - 1]) ** 2).sum(1))
    assert flagged.item() >= len(i)
    assert (got[:30] == 0).all()
    assert (np.abs(got - want) <= 0.501 * np.spacing(want.astype(np.float32))).all()


# --------------------------------------------------------------- AT energy --
@pytest.mark.parametrize("scale,finite", [(1.0, True), (3e-4, True), (1e-7, False)])
def test_at_small_products(scale, finite):
    """A regular tetrahedron: its four triplets are alike, and the last point pairs
    sum over two k at once.  At 1e-7 the products a b c are subnormal and a term
    exceeds FP32's range, so the energy is infinite."""
    x = np.array([[1, 1, 1], [1, -1, -1], [-1, 1, -1], [-1, -1, 1]], np.float64) * scale
    import torch
    t, D = tri(), dev()
    p = torch.from_numpy(x.astype(np.float32)).to(D)
    energy = torch.empty(1, dtype=torch.float64, device=D)
    ws = torch.empty(t.tet_at_workspace_size(4, 16), dtype=torch.uint8, device=D)
    t.tet_at_energy(p, energy, rho=16, workspace=ws)
    if finite:
        # equilateral side r: (1 + 3/8) / r^9 each; FP32 terms, about 20 roundings
        want = 4 * 1.375 / (np.sqrt(8.0) * np.float64(np.float32(scale))) ** 9
        assert abs(energy.item() - want) <= 2e-5 * want
    else:
        assert energy.item() == float("inf")


# ------------------------------------------- tensor-core distances, accuracy --
def _tc_edm(x, prec):
    import torch
    t, n = tri(), x.shape[0]
    out = torch.empty(n * (n + 1) // 2, device=x.device)
    ws = torch.empty(t.tri_edm_workspace_size(n, x.shape[1], prec), dtype=torch.uint8, device=x.device)
    t.tri_edm(x, out, prec=prec, workspace=ws)
    return out


def _packed64(x):
    """Packed lower triangle of distances by direct differences, in 64 bits."""
    import torch
    n, xd = x.shape[0], x.double()
    ref = torch.zeros(n, n, dtype=torch.float64, device=x.device)
    for k in range(x.shape[1]):
        df = xd[:, k, None] - xd[None, :, k]
        ref.addcmul_(df, df)
    return ref.sqrt_()[torch.tril(torch.ones_like(ref, dtype=torch.bool))]


@pytest.mark.parametrize("prec", ["BF16X6", "BF16X3"])
@pytest.mark.parametrize("n", [300, 1500])  # the second has more pairs than the list of flagged ones holds
@pytest.mark.parametrize("e", [-25, -24, -23, -22, -21, -20, -19])
def test_tc_edm_tiny_rows(prec, n, e):
    """Squares at the edge of FP32's range and below it: flagged and recomputed, so
    within 1e-5 like all others."""
    import torch
    g = torch.Generator(device=dev()).manual_seed(n)
    for d in (2, 64):
        x = (torch.randn(n, d, generator=g, device=dev()).double() * 10.0 ** e).float()
        got, ref = _tc_edm(x, getattr(tri(), prec)).double(), _packed64(x)
        assert bool(((got - ref).abs() <= 1e-5 * ref).all()), d


def test_tc_edm_recompute_rounds_as_fp64():
    """Recomputed pairs are FP64 sums rounded once: half an ulp and, for the sum's own
    rounding of at most 64 steps, 2^-24 of one."""
    import torch
    D = dev()
    for seed in range(6):
        x = 100.0 + torch.randn(1400, 64, generator=torch.Generator(device=D).manual_seed(seed), device=D)
        got, ref = _tc_edm(x, tri().BF16X3).double(), _packed64(x)
        ulp = torch.exp2(torch.floor(torch.log2(ref.clamp_min(1e-30))) - 23)
        assert bool(((got - ref).abs() <= (0.5 + 2.0 ** -24) * ulp).all()), seed


@pytest.mark.parametrize("d,most", [(224, 5.29e-6), (256, 5.23e-6), (320, 6.02e-6)])
def test_tc_edm_sum_order(d, most):
    """Uniform points, whose inner products grow with every step, so that the sums'
    truncation shows: no further off than the two-plane BF16 split that this one
    replaced, whose largest relative errors on these points are given."""
    import torch
    n = 1999
    x = torch.rand(n, d, generator=torch.Generator(device=dev()).manual_seed(1000 * d + n + 2), device=dev())
    got, ref = _tc_edm(x, tri().BF16X3).double(), _packed64(x)
    off = ref > 0
    assert float(((got - ref).abs() / ref)[off].max()) <= most
