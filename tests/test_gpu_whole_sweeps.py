"""Whole red-black sweeps (one pass per sweep, FP32 levels n >= 32): the memory that a context takes for them, and
their bits against the half-sweeps over the launch shapes they are chosen for; the corrections that follow an FMG with
boundary values on the same context."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def q():
    import paper_1201_3185_gb300 as q
    return q


def _footprint(q, n, **kw):
    """Device bytes of a context."""
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    before = torch.cuda.mem_get_info()[0]
    ctx = q.Context(n=n, nboxes=1, L0=64.0, precision=q.QUMOND_PREC_MIXED, **kw)
    took = before - torch.cuda.mem_get_info()[0]
    ctx.close()
    return took


def _black(n):
    """Bytes of the black values of a level of one set: rows padded to four entries."""
    return 4 * ((n // 2 + 1 + 3) // 4 * 4) * (n + 1) ** 2


@pytest.mark.parametrize("n,sets,without,levels", [
    # (the other context's parameters, the levels whose second black array it does not need)
    (256, 2, dict(npre=1), (256, 128, 64)),                            # odd counts run half-sweeps
    (256, 2, dict(npost=3), (256, 128, 64)),
    (128, 16, dict(bc_mode=1, rel_tol=0.0), (128,)),                   # no correction, every finest V-cycle with
                                                                       # boundary values: half-sweeps there
])
def test_second_black_arrays_only_where_whole_sweeps_run(q, n, sets, without, levels):
    kw = dict(nsets=sets, rel_tol=1e-8)
    _footprint(q, n, **kw)  # what the first context of a shape loads for good
    _footprint(q, n, **{**kw, **without})
    need = sum(_black(m) for m in levels) * sets
    # allocations come in blocks of 2 MB
    assert _footprint(q, n, **kw) - _footprint(q, n, **{**kw, **without}) >= need - 2 * (2 << 20)


def test_no_second_black_array_on_the_level_that_a_cluster_runs(q):
    # n = 32 below n = 64: its V-cycles are one kernel's (form 3) or half and whole sweeps (form 0)
    n, sets = 64, 512
    a = _footprint(q, n, nsets=sets, rel_tol=1e-8, persistent_vcycle=3)
    b = _footprint(q, n, nsets=sets, rel_tol=1e-8, persistent_vcycle=0)
    assert b - a >= _black(32) * sets - 2 * (2 << 20)


@pytest.mark.parametrize("precision,n,sets", [(1, 256, 8), (2, 256, 16)])
def test_a_context_without_room_for_the_second_black_arrays(q, precision, n, sets):
    # device memory for the context but for half of those arrays: it is created all the same, and its solves give the
    # same bits
    assert (q.QUMOND_PREC_MIXED, q.QUMOND_PREC_MIXED_FIXED) == (1, 2)
    kw = dict(n=n, nboxes=1, L0=64.0, precision=precision, nsets=sets, rel_tol=1e-8)
    g = torch.Generator(device="cuda").manual_seed(n)
    src = torch.rand(sets * (n + 1) ** 3, dtype=torch.float64, device="cuda", generator=g) - 0.5
    want, got = torch.zeros_like(src), torch.zeros_like(src)
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    ctx = q.Context(**kw)
    full = free - torch.cuda.mem_get_info()[0]
    ctx.qumond_solve_mond(0, src, None, want)
    ctx.close()
    filler = torch.empty(torch.cuda.mem_get_info()[0] - full + _black(n) * sets // 2, dtype=torch.uint8, device="cuda")
    ctx = q.Context(**kw)
    ctx.qumond_solve_mond(0, src, None, got)
    ctx.close()
    del filler
    torch.cuda.empty_cache()
    assert torch.equal(got, want)


@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("n", [4, 8, 16, 32, 64, 128])
def test_corrections_after_an_fmg_with_boundary_values(q, precision, n):
    # FMG leaves boundary values on its way up every level, and the corrections after it read zeros there: on the same
    # context the same bits as on one that never ran an FMG, from the same start
    g = torch.Generator(device="cuda").manual_seed(n)
    src = torch.rand((n + 1) ** 3, dtype=torch.float64, device="cuda", generator=g) - 0.5
    given = torch.rand_like(src) + 1.0
    kw = dict(n=n, nboxes=1, L0=64.0, precision=precision, bc_mode=q.QUMOND_BC_GIVEN, ncycle=1)
    tol = dict(rel_tol=1e-6, max_vcycles=60)
    ctx = q.Context(**kw)
    start = given.clone()
    ctx.qumond_solve_mond(0, src, None, start)
    ctx.close()
    ctx = q.Context(**kw, **tol)
    for _ in range(2):  # the second solve also follows the first's corrections
        a = given.clone()
        ctx.qumond_solve_mond(0, src, None, a)
    ctx.close()
    ctx = q.Context(**kw, **tol, warm_start=1)
    b = start.clone()
    ctx.qumond_solve_mond(0, src, None, b)
    ctx.close()
    assert torch.equal(a, b)


def _two_cycles(q, src, n, sets, **kw):
    """Two V-cycles on src from zero, on the finest level as: the FMG's own ones with zero boundary values (whole sweeps
    where they apply, from black values that are zero), the FMG's own ones with boundary values given (half-sweeps), and
    one step of the defect correction from zero (whole sweeps whose first starts from zero)."""
    kw = dict(n=n, nboxes=1, L0=64.0, precision=q.QUMOND_PREC_MIXED, nsets=sets, **kw)
    out = []
    for case in (dict(ncycle=2), dict(ncycle=2, bc_mode=q.QUMOND_BC_GIVEN),
                 dict(warm_start=1, dc_vcycles=2, max_vcycles=2, rel_tol=0.9)):
        ctx = q.Context(**kw, **case)
        phi = torch.zeros_like(src)
        ctx.qumond_solve_mond(0, src, None, phi)
        ctx.close()
        out.append(phi)
    return out


# sets: the launches of n = 32, 64, 128 take their large tiles from 2^20 groups of four entries in all sets on (273, 34
# and 5 sets), those of n = 256 with any; from n = 512 the tiles run along the rows too (2 and 4 of them)
@pytest.mark.parametrize("npre,npost", [(2, 2), (4, 2), (1, 2), (3, 1)])  # odd ones: the fallback
@pytest.mark.parametrize("n,sets", [(32, 1), (32, 280), (64, 1), (64, 34), (128, 1), (128, 8), (256, 1), (256, 2),
                                    (512, 1), (512, 2), (1024, 1)])
def test_sweeps_from_zero_give_the_bits_of_the_half_sweeps(q, n, sets, npre, npost):
    # a source that alternates along x: its full weighting is exactly zero, so FMG brings a zero to the finest level and
    # the V-cycles there start from zero in all three runs.  The coarser levels' corrections are the same launches in
    # all three, so each level's launches are compared where it is the finest
    if n == 1024 and (npre, npost) != (2, 2):
        pytest.skip("one size of four tiles along a row is enough")
    g = torch.Generator(device="cuda").manual_seed(n + sets)
    src = torch.rand(sets, n + 1, n + 1, 1, dtype=torch.float64, device="cuda", generator=g) - 0.5
    src = (src * (1.0 - 2.0 * (torch.arange(n + 1, device="cuda") % 2))).reshape(-1)
    own, given, corrected = _two_cycles(q, src, n, sets, npre=npre, npost=npost)
    assert torch.equal(own, given)
    assert torch.equal(corrected, given)
    assert torch.all(torch.isfinite(own)) and torch.any(own != 0.0)


@pytest.mark.parametrize("npre,npost", [(1, 1), (1, 2), (3, 1)])
def test_odd_counts_to_a_tolerance_give_the_bits_of_the_solve_without_allocation(q, npre, npost):
    # the half-sweeps that odd counts run, first sweeps from zero in one launch among them
    n = 64
    g = torch.Generator(device="cuda").manual_seed(npre + npost)
    src = torch.rand((n + 1) ** 3, dtype=torch.float64, device="cuda", generator=g) - 0.5
    kw = dict(n=n, nboxes=1, L0=64.0, precision=q.QUMOND_PREC_MIXED, npre=npre, npost=npost, ncycle=1, rel_tol=1e-9,
              max_vcycles=60, dc_vcycles=2)
    ctx = q.Context(**kw)
    a = torch.zeros_like(src)
    ctx.qumond_solve_mond(0, src, None, a)
    ctx.close()
    b = torch.zeros_like(src)
    q.qumond.qumond_solve_mond_noalloc(q.default_params(**kw), 0, src, None, b)
    assert torch.equal(a, b)


@pytest.mark.parametrize("npre,npost,bc,whole", [(2, 2, 0, True), (2, 4, 0, True), (1, 2, 0, False), (2, 2, 1, False)])
def test_whole_sweeps_have_a_tracer_class_of_their_own(q, npre, npost, bc, whole):
    # full multigrid on levels 128, 64, 32 (per-step form): its V-cycles, ncycle on each level, visit every level under
    # it; the restriction and the correction of a whole sweep are not counted in the classes of their own launches.
    # With boundary values given (bc 1) each level's own V-cycles are half-sweeps, the corrections under it whole ones
    n, ncycle = 128, 2
    ctx = q.Context(n=n, nboxes=1, L0=64.0, precision=q.QUMOND_PREC_MIXED, npre=npre, npost=npost, ncycle=ncycle,
                    bc_mode=bc, persistent_vcycle=0, use_graphs=0)
    src = torch.ones((n + 1) ** 3, dtype=torch.float64, device="cuda")
    phi = torch.zeros_like(src)
    ctx.qumond_trace_read(reset=True)
    ctx.qumond_solve_mond(0, src, None, phi)
    st, _, cells = ctx.qumond_trace_read(reset=True)
    ctx.close()
    count = {k: v.launches for k, v in st.items()}
    sweeps = npre + npost
    if whole:
        assert count["sweep_finest"] == ncycle * sweeps
        assert count["sweep_coarser"] == ncycle * sweeps * (2 + 3)  # 64 for itself and 128; 32 for itself, 64 and 128
        assert count["rb_half_finest"] == count["rb_half_coarser"] == count["restrict_resid_red"] == 0
        assert count["prolong_black"] == 3  # FMG's own, one a level
    elif bc == 0:
        assert count["sweep_finest"] == count["sweep_coarser"] == 0
        assert count["rb_half_finest"] > 0 and count["rb_half_coarser"] > 0
    else:
        assert count["sweep_finest"] == 0
        assert count["rb_half_finest"] == ncycle * 2 * sweeps
        assert count["sweep_coarser"] == ncycle * sweeps * (1 + 2)  # 64 for 128; 32 for 64 and 128
