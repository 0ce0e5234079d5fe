"""Kernels at the sizes where their index arithmetic can go wrong, against the oracle."""
import numpy as np
import pytest
import torch

from tests.gpu_helpers import to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def q():
    import paper_1201_3185_gb300 as q
    return q


@pytest.mark.parametrize("n,nboxes", [(4, 3), (8, 1), (16, 4)])
def test_forces_at_cell_edges(q, ora, n, nboxes):
    # points on, just inside and just outside the first and last interior cells of every box, at the centre, and
    # points that are no number: which box a point takes and its cell must be the oracle's
    L0 = 64.0
    rng = np.random.default_rng(n)
    phis = [rng.uniform(-1.0, 1.0, (n + 1) ** 3) for _ in range(nboxes)]
    axis = [0.0, -0.0, 1e-300, L0, -L0, np.nan, -np.nan, np.inf, -np.inf]
    for b in range(nboxes):
        h = L0 / 2 ** b / n
        for i in (1.0, 1.5, n / 2 + 0.25, n - 1.25, n - 1.0):
            x = -0.5 * L0 / 2 ** b + i * h
            axis += [x, np.nextafter(x, -np.inf), np.nextafter(x, np.inf)]
    pts = rng.choice(np.array(axis), size=(3, 20011))
    pts[:, :len(axis)] = axis  # the diagonal too
    ctx = q.Context(n=n, nboxes=nboxes, L0=L0)
    d = [to_dev(a) for a in pts]
    g = [torch.full_like(d[0], 7.0) for _ in range(3)]
    ctx.qumond_forces([to_dev(p) for p in phis], *d, *g)
    want = ora.forces(n, L0, (0.0, 0.0, 0.0), phis, *pts)[:3]
    # each side weights differences of values <= 1 with at most 24 rounded products and sums, times 1/(2h)
    tol = 2 * 24 * 2.0 ** -53 * 2.0 / (2.0 * L0 / 2 ** (nboxes - 1) / n)
    for a, w in zip(g, want):
        assert np.max(np.abs(a.cpu().numpy() - w)) <= tol
    ctx.close()


@pytest.mark.parametrize("n,center", [(2, 0.0), (8, 32.0), (64, -7.3), (1024, 32.0)])
def test_deposit_at_cell_edges_and_rounding_ties(q, ora, n, center):
    # coordinates on, just inside and just outside the box and cell faces (centre 32: the box starts at 0, and -0.0 is
    # in it), masses whose shares are ties, below one unit, above 2^52 (the conversion instruction) and negative
    L0, shift = 64.0, 24
    rng = np.random.default_rng(n)
    lo, h = center - 0.5 * L0, L0 / n
    axis = [0.0, -0.0, np.nan, np.inf, -np.inf, 5e-324]
    for i in (0.0, 0.5, 1.0, 1.25, n / 2, n - 1.0, n - 0.5, n):
        x = lo + i * h
        axis += [x, np.nextafter(x, -np.inf), np.nextafter(x, np.inf)]
    x, y, z = rng.choice(np.array(axis), size=(3, 4999))
    unit = 2.0 ** -shift
    m = rng.choice(np.array([0.0, 4.0, 12.0, 20.0, 1.0, 0.3, 1e-9, -4.0, -12.0, 1e6 + 0.7, 2.0 ** 52, 2.0 ** 52 - 1.0,
                             2.0 ** 53 + 2.0, 2.0 ** 40 + 0.5, -2.0 ** 54]) * unit, size=4999)
    want, _ = ora.cic_deposit(n, L0, (center,) * 3, shift, x, y, z, m)
    ctx = q.Context(n=n, nboxes=1, L0=L0, center=(center,) * 3, deposit_shift=shift)
    qf = torch.empty(ctx.nodes, dtype=torch.int64, device="cuda")
    rho = torch.empty(ctx.nodes, dtype=torch.float64, device="cuda")
    ctx.qumond_deposit(0, *(to_dev(a) for a in (x, y, z, m)), qf, rho)
    got = qf.cpu().numpy()
    assert np.array_equal(got, want)
    assert np.array_equal(rho.cpu().numpy(), got * (2.0 ** -shift * (n / L0) ** 3))
    ctx.close()


@pytest.mark.parametrize("n,sets", [(2, 1), (4, 3), (8, 1), (16, 2), (32, 1), (64, 2)])
def test_source_on_partial_tiles(q, ora, n, sets):
    # every position of the last column, row and plane within the tiles of 30 columns, 8 rows and 24 planes, several sets
    L0, a0 = 3.0 * n, 3.6
    rng = np.random.default_rng(n)
    phi = rng.uniform(-1.0, 1.0, (sets, (n + 1) ** 3))
    phi[0, :n] = 0.5  # equal neighbours: faces without a flux
    ctx = q.Context(n=n, nboxes=1, L0=L0, a0=a0, nsets=sets)
    src = torch.full((sets * (n + 1) ** 3,), 7.0, dtype=torch.float64, device="cuda")
    ctx.qumond_source(0, to_dev(phi.reshape(-1)), src)
    got = src.cpu().numpy().reshape(sets, -1)
    h = L0 / n
    # six fluxes of at most nu dPhi <= 2 + sqrt(2 a0 h), each with about ten FP32 roundings, over h^2
    tol = 60 * 2.0 ** -24 * (2.0 + np.sqrt(2.0 * a0 * h)) / h ** 2
    for s in range(sets):
        assert np.max(np.abs(got[s] - ora.source(n, h, a0, phi[s]))) <= tol
    ctx.close()


def _mond(q, src, phi0, n, box, **kw):
    ctx = q.Context(n=n, nboxes=box + 1, L0=64.0, precision=q.QUMOND_PREC_MIXED, **kw)
    phi = phi0.clone()
    ctx.qumond_solve_mond(box, src, None, phi)
    ctx.close()
    return phi


@pytest.mark.parametrize("n,sets,ncycle", [(32, 1, 2), (32, 7, 1), (64, 1, 2), (64, 5, 1), (128, 1, 1), (128, 3, 2),
                                           (256, 1, 1), (256, 2, 1), (512, 1, 1)])
def test_whole_sweeps_give_the_bits_of_the_half_sweeps(q, n, sets, ncycle):
    # full multigrid without a tolerance: with zero boundary values by bc_mode ZERO each level's V-cycles run as whole
    # sweeps, with zeros given by the caller (GIVEN) as half-sweeps, restriction and prolongation of their own
    g = torch.Generator(device="cuda").manual_seed(n + sets)
    src = torch.rand(sets * (n + 1) ** 3, dtype=torch.float64, device="cuda", generator=g) - 0.5
    phi0 = torch.zeros_like(src)
    kw = dict(ncycle=ncycle, nsets=sets)
    a = _mond(q, src, phi0, n, 0, bc_mode=q.QUMOND_BC_ZERO, **kw)
    b = _mond(q, src, phi0, n, 0, bc_mode=q.QUMOND_BC_GIVEN, **kw)
    assert torch.equal(a, b)
    if sets > 1:  # and those of the last set alone
        k = (sets - 1) * (n + 1) ** 3
        c = _mond(q, src[k:].clone(), phi0[k:].clone(), n, 0, bc_mode=q.QUMOND_BC_ZERO, ncycle=ncycle)
        assert torch.equal(a[k:], c)


def test_whole_sweeps_give_the_bits_of_the_solve_without_allocation(q):
    # that solve runs half-sweeps on every level: the corrections that start from zero are among them here
    n = 64
    g = torch.Generator(device="cuda").manual_seed(3)
    src = torch.rand((n + 1) ** 3, dtype=torch.float64, device="cuda", generator=g) - 0.5
    phi0 = torch.zeros_like(src)
    kw = dict(ncycle=1, rel_tol=1e-9, max_vcycles=40, dc_vcycles=3)
    a = _mond(q, src, phi0, n, 0, **kw)
    b = phi0.clone()
    q.qumond.qumond_solve_mond_noalloc(
        q.default_params(n=n, nboxes=1, L0=64.0, precision=q.QUMOND_PREC_MIXED, **kw), 0, src, None, b)
    assert torch.equal(a, b)


@pytest.mark.parametrize("npre,npost,ncycle", [(1, 1, 1), (2, 2, 6), (3, 1, 2)])
@pytest.mark.parametrize("n", [2, 4, 8, 16, 32])
def test_coarse_levels_match_the_oracle(q, ora, n, npre, npost, ncycle):
    # the levels that one block solves: rows of nodes in registers (n = 8, 16, FP32), a node per lane (n = 4), one
    # unknown (n = 2); boundary values given, so that each FMG level starts from values other than zero
    rng = np.random.default_rng(n + npre)
    L0 = 4.0 * n
    f = rng.uniform(-1.0, 1.0, (n + 1) ** 3)
    u = rng.uniform(-1.0, 1.0, (n + 1) ** 3)
    want = u.copy()
    ora.fmg(n, L0 / n, want, f, ncycle, npre, npost)
    for prec, tol in ((q.QUMOND_PREC_FP64, 1e-11), (q.QUMOND_PREC_MIXED, 1e-4)):
        # FP64: the same iterates, summed in another order; FP32: about 10 roundings of 2^-24 in each of at most 6
        # cycles of 4 sweeps on 5 levels, 7e-5 of the largest value if all added up
        ctx = q.Context(n=n, nboxes=1, L0=L0, precision=prec, bc_mode=q.QUMOND_BC_GIVEN, npre=npre, npost=npost,
                        ncycle=ncycle)
        phi = to_dev(u)
        ctx.qumond_solve_mond(0, to_dev(f), None, phi)
        assert np.max(np.abs(phi.cpu().numpy() - want)) <= tol * np.max(np.abs(want))
        ctx.close()


@pytest.mark.parametrize("n,ratio,sets", [(4, 2, 1), (8, 4, 2), (16, 8, 1), (64, 2, 3), (128, 4, 1)])
def test_boundary_from_the_parent(q, ora, n, ratio, sets):
    # no V-cycles to speak of: only the boundary nodes are compared; every offset of each ratio occurs
    rng = np.random.default_rng(n)
    L0 = 64.0
    par = rng.uniform(-1.0, 1.0, (sets, (n + 1) ** 3))
    ctx = q.Context(n=n, nboxes=2, L0=L0, box_ratio=ratio, nsets=sets, ncycle=1)
    phi = torch.zeros(sets * (n + 1) ** 3, dtype=torch.float64, device="cuda")
    ctx.qumond_solve_mond(1, torch.zeros_like(phi), to_dev(par.reshape(-1)), phi)
    got = phi.cpu().numpy().reshape(sets, n + 1, n + 1, n + 1)
    m = np.ones((n + 1,) * 3, dtype=bool)
    m[1:-1, 1:-1, 1:-1] = False
    for s in range(sets):
        want = np.zeros((n + 1) ** 3)
        ora.boundary_fill(n, L0, (0.0, 0.0, 0.0), par[s], L0 / ratio, (0.0, 0.0, 0.0), want)
        # exact weights, eight products of values <= 1 summed in one order: a few roundings on each side
        assert np.max(np.abs(got[s][m] - want.reshape(m.shape)[m])) <= 16 * 2.0 ** -53
    ctx.close()


@pytest.mark.parametrize("S,tensor_path", [(64, 1), (64, 0), (32, 0), (48, 1), (80, 0)])
def test_guess_gradients_on_all_tile_widths(q, S, tensor_path):
    """Levels of 64^3 to 4^3 voxels: every width of the channel tile, and weight gradients over 2048 bricks to one;
    48 and 80: levels of 24, 12, 6 and of 40, 20, 10 voxels, which no power of two divides into bricks.
    The bounds are those of the gradient test of the smaller networks (14 layers of BF16 rounding: 3 % of the whole
    vector, 15 % of a block whose terms cancel); a wrong tap, channel or voxel moves a block by tens of percent."""
    from oracle import unet as U
    from tests.test_gpu_guess import he, random_sample, rel_l2
    rng = np.random.default_rng(S)
    params = he(S)
    smp = random_sample(rng, S)
    g = q.Guess(S, 1e5)
    g.qumond_guess_set_params(to_dev(params, torch.float32))
    g.qumond_guess_tensor_path(tensor_path)
    grads = torch.empty(q.Guess.num_params(), dtype=torch.float32, device="cuda")
    g.qumond_guess_gradients([smp.cuda()], [1.0], grads)
    g.qumond_guess_status()
    got = grads.cpu().numpy().astype(np.float64)
    _, want = U.loss_and_gradients(params, [smp.float().numpy()], [1.0])
    assert rel_l2(got, want) < 3e-2
    for name, sl in U.layer_slices():
        assert rel_l2(got[sl], want[sl]) < 0.15, name
    g.close()


@pytest.mark.parametrize("n,npre,npost", [(32, 1, 2), (64, 2, 1)])
def test_fp64_coarse_levels_of_several_sets(q, n, npre, npost):
    # one cluster of blocks per set runs the levels from n = 16 down: each set's solve as if alone, bit for bit
    rng = np.random.default_rng(n)
    nodes = (n + 1) ** 3
    rhs = to_dev(rng.uniform(-1.0, 1.0, 3 * nodes))
    kw = dict(n=n, nboxes=1, L0=64.0, precision=q.QUMOND_PREC_FP64, bc_mode=q.QUMOND_BC_ZERO, npre=npre, npost=npost,
              ncycle=2)
    ctx = q.Context(nsets=3, **kw)
    phi = torch.zeros_like(rhs)
    ctx.qumond_solve_mond(0, rhs, None, phi)
    ctx.close()
    ctx = q.Context(**kw)
    for s in range(3):
        one = torch.zeros(nodes, dtype=torch.float64, device="cuda")
        ctx.qumond_solve_mond(0, rhs[s * nodes:(s + 1) * nodes].clone(), None, one)
        assert torch.equal(one, phi[s * nodes:(s + 1) * nodes])
    ctx.close()


@pytest.mark.parametrize("n", [64, 128])
def test_fp64_restriction_tiles(q, ora, n):
    # coarse grids of 31 and 63 nodes against tiles of 16 x 4 x 2: a remainder on every side
    rng = np.random.default_rng(n)
    f = rng.uniform(-1.0, 1.0, (n + 1) ** 3)
    u = rng.uniform(-1.0, 1.0, (n + 1) ** 3)
    want = u.copy()
    ora.fmg(n, 64.0 / n, want, f, 1, 1, 1)
    ctx = q.Context(n=n, nboxes=1, L0=64.0, precision=q.QUMOND_PREC_FP64, bc_mode=q.QUMOND_BC_GIVEN, npre=1, npost=1,
                    ncycle=1)
    phi = to_dev(u)
    ctx.qumond_solve_mond(0, to_dev(f), None, phi)
    # the same iterates, summed in another order
    assert np.max(np.abs(phi.cpu().numpy() - want)) <= 1e-11 * np.max(np.abs(want))
    ctx.close()
