"""Branches that a size picks: each against the path it stands beside."""
import numpy as np
import pytest
import torch

from paper_2608_16960_gb300 import synth
from paper_2608_16960_gb300.projector import Geometry, Grid, tsp_forward

pytestmark = pytest.mark.gpu


def _grid(shape, wedge=False):
    kw = dict(theta=(0.3, 2.6), phi=(0.4, 5.1)) if wedge else {}
    e = synth.grid_edges(*shape, **kw)
    return Grid.from_edges(e), e


def _geometry(kind, n_views=2, det=(19, 37)):
    if kind == "cone":
        return Geometry.cone(synth.circular_orbit(n_views, 60.0, incline_deg=20.0, phase=0.3), det, 50.0)
    if kind == "parallel":
        return Geometry.parallel(synth.random_positions(n_views, 5), det, 50.0)
    s, d = synth.random_rays(n_views * det[0] * det[1], 6)
    return Geometry.rays(torch.tensor(s, device="cuda"), torch.tensor(d, device="cuda"))


@pytest.mark.parametrize("kind", ["cone", "parallel", "rays"])
@pytest.mark.parametrize("batch", [2, 3, 4, 5, 8, 9])
def test_batched_forward_equals_each_volume(kind, batch):
    """Every number of volumes per launch: the terms of each sum are those of
    the single-volume call in the same order, so the results are the same bits."""
    grid, _ = _grid((13, 9, 22), wedge=kind == "cone")
    geom = _geometry(kind)
    rho = torch.tensor(synth.uniform_volume((batch,) + grid.shape, 3, 0.1, 1.0), device="cuda")
    y = tsp_forward(grid, geom, rho)
    for b in range(batch):
        assert torch.equal(y[b], tsp_forward(grid, geom, rho[b].contiguous()))


def _sparse(shape, pattern, seed):
    """Measurements that leave few terms per voxel (so that a lost or doubled
    lane shows), or all of them."""
    rng = np.random.default_rng(seed)
    y = rng.uniform(0.5, 1.5, shape).astype(np.float32)
    if pattern == "row":      # eight neighbouring pixels of one row: one run of lanes
        keep = np.zeros(shape, bool)
        keep[..., 5, 8:16] = True
    elif pattern == "holes":  # some lanes of each warp idle
        keep = rng.uniform(size=shape) < 0.02
    else:
        keep = np.ones(shape, bool)
    return np.where(keep, y, 0.0).astype(np.float32), int(keep.reshape(-1, *shape[-2:]).sum(axis=(0, 1, 2)).max())


# Sums of n non-negative float32 terms in any two orders differ by at most
# 2 n 2^-24 of their value; a ray meets a voxel at most four times (twice per
# half of its radial run).
def _bound(n_rays):
    return 2.0 * 4.0 * n_rays * 2.0 ** -24


@pytest.mark.parametrize("pattern", ["row", "holes", "all"])
@pytest.mark.parametrize("kind,shape", [("cone", (7, 5, 8)), ("parallel", (7, 5, 8)), ("cone", (24, 22, 44))])
@pytest.mark.parametrize("batch", [1, 2, 3, 6])
def test_combined_scatters_equal_one_add_per_segment(kind, shape, pattern, batch):
    """Coarse grids (a voxel many pixels wide: runs of lanes) and a finer one
    (pairs), odd detector sizes, idle lanes."""
    from paper_2608_16960_gb300.projector import tsp_adjoint
    grid, _ = _grid(shape)
    geom = _geometry(kind, 2, (41, 67))
    y, n = _sparse((batch,) + geom.det_shape, pattern, 5)
    y = torch.tensor(y, device="cuda")
    for tile in (4, 8, 32):
        a, b = (tsp_adjoint(grid, geom, y, launch=(128, tile, s)) for s in (0, 1))
        assert float(a.max()) > 0.0
        assert bool(((a - b).abs() <= _bound(n) * a).all())


@pytest.mark.parametrize("shape", [(7, 5, 8), (24, 22, 44)])
def test_combined_scatters_of_the_other_operators(shape):
    """Dynamic, attenuated, SIRT and batched SIRT scatters, combined against plain."""
    from paper_2608_16960_gb300.projector import (AttenuatedOperator, Batch, tsp_adjoint_dynamic, tsp_autotune_clear,
                                                  tsp_autotune_store, tsp_sirt)
    grid, _ = _grid(shape)
    geom = _geometry("cone", 2, (41, 67))
    op = AttenuatedOperator(grid, geom, (0.6, -0.4, 0.7))
    rho0 = torch.tensor(synth.uniform_volume(grid.shape, 3, 0.1, 0.3), device="cuda")
    sig0 = torch.tensor(synth.uniform_volume(grid.shape, 4, 0.2, 0.5), device="cuda")
    y = torch.tensor(_sparse(geom.det_shape, "all", 5)[0], device="cuda")
    got = []
    try:
        for s in (0, 1):
            tsp_autotune_store(grid, geom, (128, 8, 0), (128, 8, s))
            rho, sig = rho0.clone().requires_grad_(True), sig0.clone().requires_grad_(True)
            op(rho, sig).backward(y)
            x = torch.zeros(grid.shape, device="cuda")
            tsp_sirt(grid, geom, y, x, 2)
            xb = torch.zeros(grid.shape, device="cuda")
            Batch([(grid, geom, y, xb)]).sirt(2)
            got.append([tsp_adjoint_dynamic(grid, geom, y), rho.grad, sig.grad, x, xb])
    finally:
        tsp_autotune_clear()
    n = int(np.prod(geom.det_shape))
    for a, b in zip(*got):
        # gradients and iterates sum terms of both signs: against the largest entry
        assert float((a - b).abs().max()) <= _bound(n) * float(a.abs().max())


@pytest.mark.parametrize("shape,batch", [((1, 1, 32), 1), ((2, 3, 32), 1), ((3, 2, 64), 2), ((5, 7, 96), 1),
                                         ((2, 2, 128), 1), ((3, 3, 160), 1), ((2, 4, 192), 2)])
def test_network_gradients_at_the_ring_sizes(shape, batch):
    """Every azimuth count's ring of theta-rows, runs that end inside a column,
    grids of one shell and one row: each gradient entry within two bfloat16
    ulps (2^-7) of every term's two factors, doubled for the layers between,
    of the sum of its terms' magnitudes, plus 1e-4 of the layer's largest."""
    from oracle import net as onet
    from paper_2608_16960_gb300.model import WarmStartNet
    net = WarmStartNet(shape, batch)
    params = onet.init_params(3)
    rng = np.random.default_rng(4)
    params = [(w, (0.05 * rng.normal(size=b.shape)).astype(np.float32)) for w, b in params]
    net.set_params(np.concatenate([np.concatenate([w.ravel(), b.ravel()]) for w, b in params]))
    a = rng.uniform(0.0, 1.0, (batch,) + shape).astype(np.float32)
    t = rng.uniform(0.0, 1.0, (batch,) + shape).astype(np.float32)
    loss = net.loss_grad(torch.tensor(a, device="cuda"), torch.tensor(t, device="cuda"))
    got = net.get_grads()
    ref_loss, grads, operands = onet.loss_and_grads(params, a, t, keep=True)
    assert abs(loss - ref_loss) <= 1e-2 * ref_loss
    for k, (off, sh) in enumerate(net.layout()):
        ref = np.asarray(grads[k // 2][k % 2], np.float64)
        x, g = operands[k // 2]
        mags = onet.conv_wgrad(np.abs(np.asarray(x, np.float32)), np.abs(np.asarray(g, np.float32)))[k % 2]
        d = np.abs(got[off:off + ref.size].reshape(ref.shape) - ref)
        assert (d <= 2.0 ** -6 * np.asarray(mags).reshape(ref.shape) + 1e-4 * np.abs(ref).max()).all(), (k, d.max())


@pytest.mark.parametrize("kind,shape,n_views,det", [
    ("cone", (64, 48, 96), 1, (13, 9)),     # voxel rows of a few entries, a band of one detector row
    ("cone", (20, 15, 30), 2, (45, 29)),    # tens
    ("parallel", (12, 9, 20), 6, (64, 64)),  # hundreds
    ("cone", (4, 3, 6), 8, (62, 50)),       # thousands on few voxels; ray rows of a few entries
    ("polar", (20, 15, 30), 2, (30, 22)),
    ("rays", (20, 15, 30), 2, (31, 37)),
])
@pytest.mark.parametrize("batch", [1, 2, 5])
def test_lists_equal_the_traversal(kind, shape, n_views, det, batch):
    """Lane groups of every size, slices that end inside a detector, several
    volumes per pass: F and F^T from the lists against the traversal's, whose
    terms they sum in another order (non-negative: 2 n 2^-24 of the value, n
    the terms of the longest row); accumulating; without the transpose."""
    from paper_2608_16960_gb300.projector import Segments, tsp_adjoint
    grid, e = _grid(shape)
    if kind == "polar":
        geom = Geometry.polar(synth.circular_orbit(n_views, 60.0, phase=0.3), det, 50.0)
    else:
        geom = _geometry(kind, n_views, det)
    rho = torch.tensor(synth.uniform_volume((batch,) + grid.shape, 3, 0.1, 1.0), device="cuda")
    w = torch.tensor(synth.uniform_volume((batch,) + geom.det_shape, 4, 0.1, 1.0), device="cuda")
    y, g = tsp_forward(grid, geom, rho), tsp_adjoint(grid, geom, w)
    for transpose in (True, False):
        segs = Segments(grid, geom, transpose=transpose)
        off = segs.export()[0]
        n_ray = int(np.diff(off).max())
        n_vox = int(np.bincount(segs.export()[1], minlength=grid.voxels).max())
        ly = segs.forward(rho)
        assert bool(((ly - y).abs() <= 2.0 * n_ray * 2.0 ** -24 * y).all())
        lg = segs.adjoint(w)
        assert bool(((lg - g).abs() <= 2.0 * n_vox * 2.0 ** -24 * g).all())
        acc = segs.adjoint(w, out=torch.ones_like(g), accumulate=True)
        assert bool(((acc - 1.0 - g).abs() <= 2.0 * n_vox * 2.0 ** -24 * g + 2.0 ** -22 * (1.0 + g)).all())


@pytest.mark.parametrize("shells", [False, True])
@pytest.mark.parametrize("shape,nb,L", [((1, 3, 5), 4, 0), ((8, 9, 14), 5, 2), ((13, 7, 33), 6, 3), ((150, 6, 8), 9, 8)])
def test_harmonic_model_kernels(shape, nb, L, shells):
    """Shells that do not fill a tile, odd angle counts, few and many
    harmonics, the identity basis: render and its adjoint against float64
    sums over the tables (n 2^-24 of the sum of magnitudes for n terms, twice
    for the two stages)."""
    from paper_2608_16960_gb300.model import SHBSpline, ShellSH
    e = synth.grid_edges(*shape)
    m = ShellSH(e, L) if shells else SHBSpline(e, nb, L)
    B, Y = (t.astype(np.float64) for t in m.tables())
    rng = np.random.default_rng(5)
    c = rng.normal(size=m.coeff_shape).astype(np.float32)
    g = rng.normal(size=shape).astype(np.float32)
    ct = torch.tensor(c, device="cuda", requires_grad=True)
    rho = m.render(ct)
    rho.backward(torch.tensor(g, device="cuda"))
    n = 2 * (B.shape[1] + Y.shape[0] + 2) * 2.0 ** -24
    ref, mag = B @ c @ Y, np.abs(B) @ np.abs(c) @ np.abs(Y)
    assert (np.abs(rho.detach().double().cpu().numpy().reshape(ref.shape) - ref) <= n * mag).all()
    n = 2 * (B.shape[0] + Y.shape[1] + 2) * 2.0 ** -24
    G = g.reshape(shape[0], -1).astype(np.float64)
    ref, mag = B.T @ (G @ Y.T), np.abs(B.T) @ (np.abs(G) @ np.abs(Y.T))
    assert (np.abs(ct.grad.double().cpu().numpy() - ref) <= n * mag).all()


@pytest.mark.parametrize("shape,L,lam", [((1, 4, 6), 0, 0.5), ((5, 6, 10), 1, 0.0), ((18, 7, 12), 3, 2.0)])
def test_cgls_first_step_and_stops(shape, L, lam):
    """One shell and several, with and without the regulariser: a solver
    without data or without iterations returns zeros (also past the check
    every 32 iterations); its first step is alpha s with s = A^T y and alpha =
    s.s / (|A s|^2 + lam |D s|^2), A's columns from the library's own render and
    projection. Each stage sums at most N terms (rays, shells' pieces, angles,
    harmonics), so it is off by N 2^-24 of the sums of magnitudes, and alpha by
    twice the relative errors of its two norms."""
    from paper_2608_16960_gb300.model import ShellSH
    from paper_2608_16960_gb300.retrieval import Retrieval
    grid, e = _grid(shape)
    geom = Geometry.polar(synth.circular_orbit(3, 60.0, phase=0.3), (9, 11), 50.0)
    m = ShellSH(e, L)
    rng = np.random.default_rng(6)
    dev = lambda a: torch.tensor(np.asarray(a, np.float32), device="cuda")
    w, y = rng.uniform(0.5, 1.0, geom.n_rays), rng.uniform(0.5, 1.0, geom.n_rays)
    w, y = w.astype(np.float32), y.astype(np.float32)
    c, first, last = Retrieval(grid, geom, m, dev(w), dev(0 * y), lam).cgls(40)
    assert first == 0.0 and last == 0.0 and not bool(c.any())
    solver = Retrieval(grid, geom, m, dev(w), dev(y), lam)
    w, y = w.astype(np.float64), y.astype(np.float64)
    c, first, last = solver.cgls(0)
    assert not bool(c.any()) and abs(first - y @ y) <= 1e-12 * (y @ y) and last == first
    nc = shape[0] * m.nq
    A = np.zeros((geom.n_rays, nc))
    M = np.zeros((nc, geom.n_rays))  # |A| from the magnitudes of the basis
    for j in range(nc):
        cj = np.zeros(nc)
        cj[j] = 1.0
        rho = m.render(dev(cj.reshape(m.coeff_shape)))
        A[:, j] = w * tsp_forward(grid, geom, rho).double().cpu().numpy().reshape(-1)
        M[j] = w * tsp_forward(grid, geom, rho.abs()).double().cpu().numpy().reshape(-1)
    c, first, last = solver.cgls(1)
    s, Du = A.T @ y, np.diff(np.eye(shape[0]), axis=0)
    D = np.kron(Du, np.eye(m.nq))
    N = 2 * (geom.n_rays + 2 * sum(shape) + shape[1] * shape[2] + m.nq) * 2.0 ** -24
    ds, As, Ds = N * (M @ y), A @ s, D @ s
    den = As @ As + lam * Ds @ Ds
    dden = np.linalg.norm(M.T @ (ds + N * np.abs(s))) + np.sqrt(lam) * np.linalg.norm(np.abs(D) @ (ds + N * np.abs(s)))
    rel = 2 * np.linalg.norm(ds) / np.linalg.norm(s) + 2 * dden / np.sqrt(den)
    x = s @ s / den * s
    got = c.double().cpu().numpy().reshape(-1)
    assert np.linalg.norm(got - x) <= 2 * (rel * np.linalg.norm(x) + s @ s / den * np.linalg.norm(ds))


@pytest.mark.parametrize("need_sigma,need_tau1", [(True, True), (True, False), (False, True), (False, False)])
@pytest.mark.parametrize("shape,det", [((9, 8, 12), (40, 40)), ((20, 15, 30), (256, 256))])
def test_attenuated_gradients_overwritten_and_added(shape, det, need_sigma, need_tau1):
    """Gradients that are overwritten (sums scattered, the voxel's factors
    applied once) against the same added to zeros (the factors in every
    segment's terms), for each set of outputs, with lanes combined and not;
    voxels that no ray crosses stay zero at an infinite density. Terms of one
    sign each (rays' weights are positive), so with n terms a voxel each form
    is off by (n + 8) 2^-24 of the sums of magnitudes: |g_tau1| / rho and
    |g_sigma| sigma / rho for rho's two parts."""
    from paper_2608_16960_gb300.projector import (Segments, atten_backward, atten_forward, optical_depth_adjoint,
                                                  sunward_geometry)
    grid, e = _grid(shape)
    geom = Geometry.cone(synth.circular_orbit(2, 60.0, phase=0.3), det, 8.0)  # misses the outer voxels
    sun = sunward_geometry(grid, [1.0, 0.4, 0.2])
    off, vox, _ = Segments(grid, geom, transpose=False).export()
    hits = np.bincount(vox, minlength=grid.voxels)
    dev = lambda a: torch.tensor(a, device="cuda")
    rho = synth.uniform_volume(grid.shape, 3, 0.1, 1.0)
    rho.reshape(-1)[hits == 0] = np.inf
    sigma = synth.uniform_volume(grid.shape, 4, 0.01, 0.02)
    tau1 = synth.uniform_volume(grid.shape, 5, 0.1, 0.5)
    w = synth.uniform_volume(geom.det_shape, 6, 0.5, 1.0)
    rho, sigma, tau1, w = dev(rho), dev(sigma), dev(tau1), dev(w)
    y = atten_forward(grid, geom, rho, sigma, tau1)
    full = atten_backward(grid, geom, rho, sigma, tau1, y, w, out=tuple(torch.zeros_like(rho) for _ in range(3)),
                          accumulate=True)
    mag = (full[2].double().abs() / rho.double() + full[1].double().abs() * sigma.double() / rho.double()).cpu().numpy()
    mag = [np.nan_to_num(mag.reshape(-1), nan=0.0)] + [full[k].double().abs().cpu().numpy().reshape(-1) for k in (1, 2)]
    got = atten_backward(grid, geom, rho, sigma, tau1, y, w, need_sigma=need_sigma, need_tau1=need_tau1)
    assert (got[1] is None) == (not need_sigma) and (got[2] is None) == (not need_tau1)
    for k in range(3):
        if got[k] is None:
            continue
        a, b = (t.double().cpu().numpy().reshape(-1) for t in (got[k], full[k]))
        assert (a[hits == 0] == 0.0).all()
        assert (np.abs(a - b) <= 2.0 * (hits + 8) * 2.0 ** -24 * mag[k])[hits > 0].all()
    soff, svox, _ = Segments(grid, sun, transpose=False).export()
    shits = np.bincount(svox, minlength=grid.voxels).reshape(grid.shape)
    rho = dev(synth.uniform_volume(grid.shape, 3, 0.1, 1.0))
    gt = dev(synth.uniform_volume(grid.shape, 7, 0.5, 1.0))
    full = optical_depth_adjoint(grid, sun, rho, sigma, gt, out=(torch.zeros_like(rho), torch.zeros_like(rho)),
                                 accumulate=True)
    got = optical_depth_adjoint(grid, sun, rho, sigma, gt, need_sigma=need_sigma)
    for a, b in zip(got, full):
        if a is not None:
            b = b.double().cpu().numpy()
            assert (np.abs(a.double().cpu().numpy() - b) <= 2.0 * (shits + 8) * 2.0 ** -24 * np.abs(b)).all()


@pytest.mark.parametrize("shape,batch", [((1, 1, 32), 1), ((2, 9, 32), 1), ((3, 7, 64), 1), ((2, 5, 96), 2),
                                         ((2, 3, 160), 1), ((2, 3, 192), 1)])
def test_one_channel_weight_gradients_keep_float32(shape, batch):
    """Partial tiles of theta-rows at each azimuth count. With centre taps of
    powers of two and nothing in the layers between, every operand is exact
    but for the residual's own rounding (2^-23 of it), so the one-channel
    layers' weight gradients show the sums' error alone: at most 9 matrix
    steps a tile, one addition a tile, 8 warps and 42 rows of partial sums, each
    within 2^-22 of the sum of the terms' magnitudes (64 in all)."""
    from oracle import net as onet
    from paper_2608_16960_gb300.model import WarmStartNet
    net = WarmStartNet(shape, batch)
    params = [(np.zeros_like(w), np.zeros_like(b)) for w, b in onet.init_params(3)]
    params[0][0][13, :, 0] = 2.0 ** -(np.arange(32) % 4)
    params[5][0][13, 0, :4] = 2.0 ** -np.arange(4)
    net.set_params(np.concatenate([np.concatenate([w.ravel(), b.ravel()]) for w, b in params]))
    rng = np.random.default_rng(4)
    a = rng.integers(0, 200, (batch,) + shape).astype(np.float32) / 128
    t = rng.uniform(0.0, 3.0, a.shape).astype(np.float32)
    net.loss_grad(torch.tensor(a, device="cuda"), torch.tensor(t, device="cuda"))
    got = net.get_grads()
    _, grads, operands = onet.loss_and_grads(params, a, t, keep=True)
    for layer in (0, 5):
        x, g = operands[layer]
        mags = onet.conv_wgrad(np.abs(np.asarray(x, np.float32)), np.abs(np.asarray(g, np.float32)))
        for k in range(2):
            off, sh = net.layout()[2 * layer + k]
            ref = np.asarray(grads[layer][k], np.float64).reshape(sh)
            d = np.abs(got[off:off + ref.size].reshape(sh) - ref)
            assert (d <= 64 * 2.0 ** -22 * np.asarray(mags[k]).reshape(sh)).all(), (layer, k, d.max())


@pytest.mark.parametrize("nr,L", [(3, 0), (33, 8)])
def test_render_transpose_keeps_small_partial_sums(nr, L):
    """A shell's sum over 256 angles: seven of eight runs of 32 sum to 0.45 ulp
    of the first's, so that adding them to it one by one in float32 loses 3
    ulps. Within a run the terms are equal and their sums exact, so what
    remains is each product's rounding and the last one: 2^-23 of the value."""
    from paper_2608_16960_gb300.model import ShellSH
    e = synth.grid_edges(nr, 16, 16)
    m = ShellSH(e, L)
    y0 = m.tables()[1][0]
    assert (y0 == y0[0]).all()
    small = 0.45 * np.spacing(np.float32(32) * y0[0]) / (32 * y0[0])
    g = np.full((nr, 256), small, np.float32)
    g[:, :32] = 1.0
    c = torch.zeros(m.coeff_shape, device="cuda", requires_grad=True)
    m.render(c).backward(torch.tensor(g.reshape(nr, 16, 16), device="cuda"))
    got = c.grad[:, 0].double().cpu().numpy()
    ref = (g.astype(np.float64) * np.float64(y0[0])).sum(1)
    assert (np.abs(got - ref) <= 2.0 ** -23 * ref).all(), (got - ref) / ref


@pytest.mark.parametrize("kind", ["cone", "parallel"])
def test_rays_aimed_at_the_origin(kind):
    """The centre pixel of an odd detector: the line passes the origin at the
    rounding residue of its set-up, anywhere from zero to 1e-13, and its polar
    and azimuth indices jump there, inside the innermost sphere. Each ray within
    the parity rule of the oracle's."""
    import oracle
    from _util import parity
    grid, e = _grid((20, 16, 31))
    pos = [synth.random_positions(400, 5)]
    pos += [synth.circular_orbit(1000, 60.0, incline_deg=a, phase=0.3) for a in (1.0, 5.0, 20.0)]
    pos = np.concatenate(pos)
    rho = synth.uniform_volume(grid.shape, 3, 0.1, 1.0)
    if kind == "cone":
        geom, rays = Geometry.cone(pos, (1, 1), 5.0), oracle.cone_rays(pos, 1, 1, 5.0)
    else:
        geom, rays = Geometry.parallel(pos, (1, 1), 5.0), oracle.parallel_rays(pos, 1, 1, 5.0)
    y = tsp_forward(grid, geom, torch.tensor(rho, device="cuda")).cpu().numpy()
    parity(y, oracle.forward(e, *rays, rho), what=f"{kind} rays aimed at the origin")


@pytest.mark.parametrize("k", [-60, -20, 7, 40])
def test_units_of_length(k):
    """Grid and views in a unit 2^-k times the other's: the same lengths times
    2^k, exactly (a grid whose squared radii approach the smallest floats too)."""
    e = synth.grid_edges(20, 15, 30)
    pos = synth.circular_orbit(3, 60.0, incline_deg=20.0, phase=0.3)
    rho = torch.tensor(synth.uniform_volume((20, 15, 30), 3, 0.1, 1.0), device="cuda")
    a = tsp_forward(Grid.from_edges(e), Geometry.cone(pos, (33, 35), 50.0), rho)
    s = 2.0 ** k
    b = tsp_forward(Grid(e.r * s, e.theta, e.phi), Geometry.cone(pos * s, (33, 35), 50.0), rho)
    assert float(a.max()) > 0.0 and torch.equal(b / s, a)


def test_bias_gradients_of_long_rows_of_partial_sums():
    """A large value at the start of every multiprocessor's share of the rows
    and then ones that a running float32 sum of it rounds, each by the same
    2^-7: 430 of them a thread would lose 6e-6 of the sum. Every gradient value
    is exact in bfloat16 (pass-through layers, a power-of-two mean), so what
    remains is the sums' rounding: at most 2 plain additions a row, one
    remainder, 3 shuffles, 4 warps, 8 rows of partial sums and the last
    addition, 20 ulps in all."""
    from oracle import net as onet
    from paper_2608_16960_gb300.model import WarmStartNet
    batch, shape = 8, (64, 64, 64)
    net = WarmStartNet(shape, batch)
    params = [(np.zeros_like(w), np.full_like(b, 2.0 ** -10)) for w, b in onet.init_params(3)]
    params[5][0][13, 0, :] = (-1.0) ** np.arange(32)
    params[5][1][:] = 0.0
    net.set_params(np.concatenate([np.concatenate([w.ravel(), b.ravel()]) for w, b in params]))
    rows, n = batch * shape[0] * shape[1], batch * int(np.prod(shape))
    g = np.full((rows, shape[2]), 1.0 + 2.0 ** -7)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    g[rows * np.arange(sms) // sms] = 2.0 ** 18
    t = torch.tensor((-g * (n / 2)).astype(np.float32).reshape((batch,) + shape), device="cuda")
    net.loss_grad(torch.zeros_like(t), t)
    got = net.get_grads()
    for layer in (1, 2, 3, 4):
        off, sh = net.layout()[2 * layer + 1]
        ref = g.sum() * (-1.0) ** np.arange(32)
        assert (np.abs(got[off:off + 32] - ref) <= 20 * 2.0 ** -24 * np.abs(ref)).all(), layer


def test_attenuated_density_gradient_of_cancelling_terms():
    """One voxel, 4096 times the same ray: each ray's two terms of the density
    gradient cancel to a thousandth, so the sum of their small remainders has
    to be that of one ray times 4096, within the rounding of 4096 additions
    (2^-24 of the sum each), not that of either term's."""
    from paper_2608_16960_gb300.projector import atten_backward, atten_forward
    grid = Grid(np.array([0.0, 2.0]), np.array([0.0, np.pi]), np.array([0.0, 2.0 * np.pi]))
    chord, full = 2.0 * np.sqrt(4.0 - 0.3 ** 2 - 0.4 ** 2), lambda v: torch.full((1, 1, 1), v, device="cuda")
    rho, sigma, tau1 = full(0.5), full(1.001 / (0.5 * chord)), full(0.2)
    got = []
    for n in (1, 4096):
        x, d = (torch.tensor(v, device="cuda").reshape(3, 1).repeat(1, n) for v in ([-5.0, 0.3, 0.4], [1.0, 0.0, 0.0]))
        geom = Geometry.rays(x, d)
        y = atten_forward(grid, geom, rho, sigma, tau1)
        got.append(float(atten_backward(grid, geom, rho, sigma, tau1, y, torch.ones(n, device="cuda"))[0]))
    assert 0.0 < abs(got[0]) < 0.01
    assert abs(got[1] - 4096 * got[0]) <= 4096 * 2.0 ** -24 * abs(4096 * got[0]), got


@pytest.mark.parametrize("fov,empty", [(0.02, False), (8.0, True)])
def test_lists_of_a_large_grid_that_few_rays_meet(fov, empty):
    """Voxel offsets of 64 M voxels of which next to none have entries: right,
    and written by all of the GPU (under 20 ms; one thread over the gap takes
    hundreds)."""
    import time
    from paper_2608_16960_gb300.projector import Segments
    grid, _ = _grid((250, 256, 1000))
    pos = synth.circular_orbit(1, 60.0, incline_deg=20.0, phase=0.3)
    geom = Geometry.cone(pos, (8, 8), fov, look_at=2.0 * pos if empty else None)
    ts = []
    for _ in range(4):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        s = Segments(grid, geom)
        torch.cuda.synchronize()
        ts.append(time.perf_counter() - t0)
    t = min(ts)
    off, vox, _ = s.export()
    assert (off[-1] == 0) == empty
    voff = s.export_transposed()[0]
    assert np.array_equal(np.diff(voff), np.bincount(vox, minlength=grid.voxels))
    assert t < 0.02, t


@pytest.mark.parametrize("shape,n_views,det", [((4, 3, 6), 8, (62, 50)),       # one pass of the sort by voxel
                                               ((20, 15, 30), 3, (45, 29)),    # two
                                               ((64, 48, 96), 2, (61, 37)),    # three
                                               ((260, 256, 256), 1, (23, 21))])  # four
@pytest.mark.parametrize("kind", ["cone", "rays"])
def test_lists_built_in_little_memory(shape, n_views, det, kind):
    """A build that may not take its usual scratch: the sort in the lists' own
    place and the rows filled in pieces give the same lists, and without the
    transpose no scratch grows with the segments at all."""
    from paper_2608_16960_gb300._lib import TspError, load
    from paper_2608_16960_gb300.projector import Segments
    grid, _ = _grid(shape)
    geom = _geometry(kind, n_views, det)
    L = load()
    a = Segments(grid, geom)
    plain, columns = a.export(), a.export_transposed()
    rho = torch.tensor(synth.uniform_volume(grid.shape, 3, 0.1, 1.0), device="cuda")
    y = a.forward(rho)
    S, V = int(plain[0][-1]), grid.voxels
    tiles = -(-S // 2048)
    passes = -(-max(1, (V - 1).bit_length()) // 8)
    need = 4 * (1, 3, 2, 3)[passes - 1] * S + 256 * tiles * 12 + 4 * V + 8 * (max(256 * tiles, V) // 2048) + 4096
    try:
        for block in (-1, 0):
            assert L.tsp_debug_segments_memory(block, need) == 0
            b = Segments(grid, geom)
            for u, v in zip(plain + columns, b.export() + b.export_transposed()):
                assert np.array_equal(u, v)
            assert torch.equal(b.forward(rho), y)
            assert L.tsp_debug_segments_memory(block, need - 2 * S) == 0
            with pytest.raises(TspError) as e:
                Segments(grid, geom)
            assert e.value.status == 3  # TSP_ENOMEM
            for most in (8 * S // 5, 0):
                assert L.tsp_debug_segments_memory(block, most) == 0
                c = Segments(grid, geom, transpose=False)
                for u, v in zip(plain, c.export()):
                    assert np.array_equal(u, v)
                assert torch.equal(c.forward(rho), y)
    finally:
        L.tsp_debug_segments_memory(-1, -1)


@pytest.mark.parametrize("transpose", [True, False])
@pytest.mark.parametrize("limit", [-1, 1])
def test_build_out_of_memory_between_single_allocations(transpose, limit):
    """Lists too large for one block take an allocation an array: whichever of
    them fails, with the usual scratch or without, the build returns
    TSP_ENOMEM, frees the ones before it, and the next build succeeds."""
    import ctypes
    from paper_2608_16960_gb300._lib import TspError, load
    from paper_2608_16960_gb300.projector import Segments, tsp_device_status
    grid, _ = _grid((10, 8, 12))
    geom = _geometry("cone", 2, (24, 24))
    L = load()
    count = ctypes.c_int64()

    def allocations():
        assert L.tsp_debug_allocation_count(ctypes.byref(count)) == 0
        return count.value

    ref = Segments(grid, geom, transpose=transpose)
    S, V = int(ref.export()[0][-1]), grid.voxels
    tiles = -(-S // 2048)
    # the transposed build without its scratch of 16 bytes a segment: 12 and what does not grow by segment
    need = 12 * S + 256 * tiles * 12 + 4 * V + 8 * (max(256 * tiles, V) // 2048) + 4096
    scratch = -1 if limit < 0 else (need if transpose else 0)
    rho = torch.tensor(synth.uniform_volume(grid.shape, 3, 0.1, 1.0), device="cuda")
    y = ref.forward(rho)
    try:
        assert L.tsp_debug_segments_memory(0, scratch) == 0
        n0 = allocations()
        assert torch.equal(Segments(grid, geom, transpose=transpose).forward(rho), y)
        n = allocations() - n0
        assert n >= (18 if transpose else 8)
        torch.cuda.synchronize()
        free0 = torch.cuda.mem_get_info()[0]
        for k in range(n):
            assert L.tsp_debug_fail_allocation(k) == 0
            before = allocations()
            with pytest.raises(TspError) as e:
                Segments(grid, geom, transpose=transpose)
            assert e.value.status == 3 and allocations() - before == k + 1  # it stopped at the one that failed
            assert torch.equal(Segments(grid, geom, transpose=transpose).forward(rho), y)
    finally:
        L.tsp_debug_fail_allocation(-1)
        L.tsp_debug_segments_memory(-1, -1)
    torch.cuda.synchronize()
    assert torch.cuda.mem_get_info()[0] >= free0 - (64 << 20)
    assert tsp_device_status() == 0


def test_chunked_workspace_after_out_of_memory():
    """The SIRT workspace fails to be allocated once while the builds' scratch
    is kept for the next item: the driver gives that back and tries again, and
    every item ends as without the failure."""
    import ctypes
    from paper_2608_16960_gb300._lib import load
    from paper_2608_16960_gb300.projector import Segments, sirt_chunked, tsp_device_status
    L = load()
    count = ctypes.c_int64()
    items, per_item = [], 0
    for k in range(2):
        grid, _ = _grid((8 + 2 * k, 6 + k, 12 + 4 * k))
        geom = _geometry("cone", 2, (24, 24))
        y = torch.tensor(synth.uniform_volume(geom.det_shape, 7 + k, 0.5, 1.0), device="cuda")
        items.append((grid, geom, y))
        L.tsp_debug_allocation_count(ctypes.byref(count))
        n0 = count.value
        Segments(grid, geom)
        L.tsp_debug_allocation_count(ctypes.byref(count))
        per_item += count.value - n0
    runs = []
    try:
        for fail_at in (-1, per_item):
            xs = [(g, m, y, torch.zeros(g.shape, device="cuda")) for g, m, y in items]
            L.tsp_debug_fail_allocation(fail_at)
            sirt_chunked(xs, 3, budget_bytes=1 << 40)
            runs.append([x[3] for x in xs])
    finally:
        L.tsp_debug_fail_allocation(-1)
    for a, b in zip(*runs):
        assert torch.equal(a, b)
    assert tsp_device_status() == 0


@pytest.mark.parametrize("kind,n_views,det", [("cone", 5, (1001, 997)), ("parallel", 2, (3, 1 << 20)), ("cone", 12, (2, 2)),
                                              ("rays", 3, (700, 701))])
def test_export_of_many_rays(kind, n_views, det):
    """Pieces of rays that begin and end anywhere in a view, a detector's band
    longer than a piece, rays without entries: the export gives the rays'
    lists as counted and summed by the walk, at a copy's speed (under 3 ns an
    entry, 20 ms at least; a host loop takes 6 to 8)."""
    import time
    from paper_2608_16960_gb300.projector import Segments, tsp_count_segments
    grid, _ = _grid((12, 9, 14))
    geom = _geometry(kind, n_views, det)
    segs = Segments(grid, geom, transpose=False)
    rho = torch.tensor(synth.uniform_volume(grid.shape, 3, 0.1, 1.0), device="cuda")
    ts = []
    for _ in range(3):
        t0 = time.perf_counter()
        off, vox, ln = segs.export()
        ts.append(time.perf_counter() - t0)
    t = min(ts)
    assert np.array_equal(np.diff(off), tsp_count_segments(grid, geom).cpu().numpy().reshape(-1))
    y = np.concatenate([[0.0], np.cumsum(rho.cpu().numpy().reshape(-1).astype(np.float64)[vox] * ln)])
    y = y[off[1:]] - y[off[:-1]]
    ref = tsp_forward(grid, geom, rho).double().cpu().numpy().reshape(-1)
    assert np.abs(y - ref).max() <= 1e-5 * ref.max()
    assert t <= max(3e-9 * len(vox), 0.02), (t, len(vox))


@pytest.mark.parametrize("shape,n_views,det,dynamic", [((60, 36, 72), 1, 257, False), ((80, 45, 90), 1, 300, False),
                                                      ((40, 30, 60), 4, 181, True)])
def test_scatters_of_few_rays_are_not_combined_at_a_loss(shape, n_views, det, dynamic):
    """Wide voxels, but few rays on a fine grid: the untuned adjoint takes no
    longer than one add per segment (5% for the clock; combined it takes 8 to 23% longer)."""
    from paper_2608_16960_gb300.projector import (tsp_adjoint, tsp_adjoint_dynamic, tsp_autotune_clear,
                                                  tsp_autotune_store)
    grid, _ = _grid(shape)
    geom = _geometry("cone", n_views, (det, det))
    y = torch.rand(geom.det_shape, device="cuda")
    out = torch.empty(((n_views,) if dynamic else ()) + grid.shape, device="cuda")
    call = (lambda: tsp_adjoint_dynamic(grid, geom, y, out)) if dynamic else (lambda: tsp_adjoint(grid, geom, y, out))

    def time():
        for _ in range(10):
            call()
        torch.cuda.synchronize()
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(50):
            call()
        b.record()
        b.synchronize()
        return a.elapsed_time(b)

    untuned, plain = [], []
    try:
        for _ in range(3):
            tsp_autotune_clear()
            untuned.append(time())
            tsp_autotune_store(grid, geom, (128, 8, 0), (128, 8, 0))
            plain.append(time())
    finally:
        tsp_autotune_clear()
    assert min(untuned) <= 1.05 * min(plain), (untuned, plain)


def test_network_gradients_of_an_infinite_input():
    """One infinite voxel, everything positive, the reach of all layers inside
    the grid: activations, output and gradients around it are +inf, so every
    weight's and bias's gradient is a sum of positive terms of which some are
    infinite: +inf, not NaN."""
    from oracle import net as onet
    from paper_2608_16960_gb300.model import WarmStartNet
    shape = (32, 32, 32)
    net = WarmStartNet(shape, 1)
    params = [(np.full_like(w, 1.0 / 1024), np.full_like(b, 0.01)) for w, b in onet.init_params(3)]
    net.set_params(np.concatenate([np.concatenate([w.ravel(), b.ravel()]) for w, b in params]))
    a = torch.full((1,) + shape, 0.5, device="cuda")
    a[0, 16, 16, 16] = float("inf")
    loss = net.loss_grad(a, torch.zeros_like(a))
    got = net.get_grads()
    assert loss == np.inf
    for k, (off, sh) in enumerate(net.layout()):
        assert (got[off:off + int(np.prod(sh))] == np.inf).all(), k


@pytest.mark.parametrize("na", [32, 64, 96, 128, 160, 192])
def test_network_gradients_across_the_azimuth_wrap(na):
    """Input and gradient at azimuths 0 and N_a - 1 alone: the taps da = -1 and
    +1 of the weight gradients then consist of the wrapped terms, which the ring
    slots' copies hold by a patch of their own. Layers that pass their input
    through (zero weights; biases of 2^-20, which open the masks and are lost in
    bfloat16 beside an input), powers of two for operands: every product is
    exact, and the sums of at most 64 terms are held to 2^-16 of their
    magnitudes' (64 additions cut off at 2^-23 each, four times over)."""
    from oracle import net as onet
    from paper_2608_16960_gb300.model import WarmStartNet
    shape, batch = (4, 8, na), 1
    net = WarmStartNet(shape, batch)
    params = [(np.zeros_like(w), np.full_like(b, 2.0 ** -20)) for w, b in onet.init_params(3)]
    params[0][0][13, :, 0] = 2.0 ** -(np.arange(32) % 4)
    params[0][1][:] = 0.0
    params[5][0][13, 0, :] = 2.0 ** -(np.arange(32) % 3)
    params[5][1][:] = 0.0
    net.set_params(np.concatenate([np.concatenate([w.ravel(), b.ravel()]) for w, b in params]))
    rng = np.random.default_rng(4)
    a = np.zeros((batch,) + shape, np.float32)
    a[..., [0, na - 1]] = 2.0 ** rng.integers(-2, 3, (batch,) + shape[:2] + (2,))
    # the target that leaves a gradient of powers of two there and none elsewhere
    out = net.forward(torch.tensor(a, device="cuda")).cpu().numpy()
    g = np.zeros_like(a)
    g[..., [0, na - 1]] = 2.0 ** rng.integers(-2, 3, (batch,) + shape[:2] + (2,))
    net.loss_grad(torch.tensor(a, device="cuda"), torch.tensor(out - g, device="cuda"))
    got = net.get_grads()
    x0 = a[..., None].astype(np.float64) * params[0][0][13, :, 0]
    mean = float(torch.tensor(np.float32(2.0 / a.size)).bfloat16())
    gz = mean * g[..., None].astype(np.float64) * params[5][0][13, 0]

    def shift(x, o):
        z = np.roll(x, (-o[0], -o[1], -o[2]), (1, 2, 3))
        for d in (0, 1):
            if o[d]:
                idx = [slice(None)] * z.ndim
                idx[d + 1] = -1 if o[d] > 0 else 0
                z[tuple(idx)] = 0.0
        return z

    for layer in (1, 2, 3, 4):
        off, sh = net.layout()[2 * layer]
        dw = got[off:off + 27 * 32 * 32].reshape(27, 32, 32)
        for tap in range(27):
            o = (tap // 9 - 1, tap // 3 % 3 - 1, tap % 3 - 1)
            xs = shift(np.where(x0 > 0.0, x0, (layer - 1) * 2.0 ** -20), o).reshape(-1, 32)
            ref = gz.reshape(-1, 32).T @ xs
            assert (ref > 2.0 ** -12 * gz.max()).all()
            assert (np.abs(dw[tap] - ref) <= 2.0 ** -16 * ref).all(), (layer, tap, np.abs(dw[tap] / ref - 1.0).max())


def test_lists_of_one_handle_on_two_streams():
    """Forward and adjoint calls on one handle enqueued on two streams at once
    share nothing but the lists: each result is that of the call by itself."""
    from paper_2608_16960_gb300.projector import Segments
    grid, _ = _grid((30, 24, 48))
    geom = _geometry("cone", 8, (128, 128))
    segs = Segments(grid, geom)
    rho = [torch.tensor(synth.uniform_volume((b,) + grid.shape, 3 + b, 0.1, 1.0), device="cuda") for b in (1, 3)]
    w = [torch.tensor(synth.uniform_volume((b,) + geom.det_shape, 5 + b, 0.1, 1.0), device="cuda") for b in (1, 3)]
    alone = [(segs.forward(r), segs.adjoint(v)) for r, v in zip(rho, w)]
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in range(2)]
    got = [[], []]
    for _ in range(20):
        for k, st in enumerate(streams):
            with torch.cuda.stream(st):
                got[k].append((segs.forward(rho[k]), segs.adjoint(w[k])))
    torch.cuda.synchronize()
    for k in range(2):
        for y, g in got[k]:
            assert torch.equal(y, alone[k][0]) and torch.equal(g, alone[k][1])
