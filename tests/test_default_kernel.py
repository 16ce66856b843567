"""The default cell kernels (tile configuration 0: line kernels, one-launch assembly) against the oracle
at the sizes where their tiles, column forms and assembly can go wrong.

* Column counts: one column (a tile holds several cells), counts below, at and above a
  tile of every degree, odd counts (no 8-byte rows), counts that leave a partial tile;
  real and complex, with the staged (16-byte rows) and the unstaged gather.
* Axis-aligned cells (per-cell scalars) and jittered ones (per-point coefficients).
* n_q = n_p + 2, the scaled form, and projectors on cells of several column tiles.
* The one-launch assembly gives the same bits twice, in every precision, and the bits of the
  colour-by-colour scatter (which a stream other than the set-up one takes for an operator
  without projectors).
* The same with projectors, in the small, flat and wide forms, and in the filter's accumulating
  applications (contexts set up without slots go colour by colour).
* Applications of one context in both storage widths may overlap.

Tolerances as in test_parity_apply: 1e-12 for FP64 and pairs of floats, 1e-5 for FP32, per
column and per entry.
"""
import dataclasses

import numpy as np
import pytest

from paper_2512_08571_gb300 import fe_ks as fk
from synth.host_problem import HostProblem
from oracle.operator import Problem
from synth import Workload, trial_vectors
from gpu_util import gpu_apply, parity_err, round_input, torch_dtype

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = {fk.FE_KS_F64: 1e-12, fk.FE_KS_F32: 1e-5, fk.FE_KS_F64E: 1e-12}
PREC = [fk.FE_KS_F64, fk.FE_KS_F32, fk.FE_KS_F64E]
COLUMNS = (1, 2, 3, 7, 8, 12, 19, 32, 33)   # tiles hold 4..32 FP32 columns, 2..16 FP64 ones


def _wl(p, cplx, jitter, nqx=0, n=2, n_atoms=2, n_v=max(COLUMNS)):
    return Workload(f"line{p}{cplx}{jitter}", L=4.0 * n / 2, n=n, p=p, nq=p + 1 + nqx, n_v=n_v, jitter=jitter, gga=True,
                    kfrac=(0.2, 0.1, -0.3) if cplx else (0.0, 0.0, 0.0), complex=cplx, n_atoms=n_atoms, seed=7700 + p)


@pytest.mark.parametrize("jitter", [0.0, 0.08])
@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("p", [1, 2, 3, 4, 5, 6, 7, 8])
def test_columns_and_degrees(p, cplx, jitter):
    wl = _wl(p, cplx, jitter, n=3 if p < 3 else 2)
    hp, X = HostProblem(wl), trial_vectors(wl)
    P = Problem(wl)
    Yref64, Yref32 = P.apply(X), P.apply(round_input(X, fk.FE_KS_F32))
    for precision in PREC:
        for nv in COLUMNS:
            Y = gpu_apply(hp, np.ascontiguousarray(round_input(X, precision)[:, :nv]), precision)
            ref = (Yref32 if precision == fk.FE_KS_F32 else Yref64)[:, :nv]
            assert parity_err(Y, ref) <= TOL[precision], (precision, nv)


@pytest.mark.parametrize("jitter", [0.0, 0.08])
@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("p", [1, 2, 3, 4, 5, 6, 7, 8])
def test_full_tiles(p, cplx, jitter):
    """As many columns as give every multiprocessor one full tile (the kernels take tiles of two
    elements below that), less a few so that the last tile of a cell is partial and, for real
    FP32, rows are not 8-byte aligned; the FP32 case runs the wide form (a block per cell)."""
    n = 3 if p < 3 else 2
    vg = 16 if p < 4 else 8 if p < 6 else 4
    vgf = 8 if p == 6 else vg     # pairs of floats
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    elems = sms * vg // n ** 3 - 1
    cols = {fk.FE_KS_F64: elems, fk.FE_KS_F64E: sms * vgf // n ** 3 - 1, fk.FE_KS_F32: 2 * elems - (0 if cplx else 1)}
    nvs = {k: v // 2 if cplx else v for k, v in cols.items()}
    wl = _wl(p, cplx, jitter, n=n, n_v=max(nvs.values()))
    hp, X = HostProblem(wl), trial_vectors(wl)
    P = Problem(wl)
    ref = P.apply(X)
    for precision in PREC:
        Xin = np.ascontiguousarray(round_input(X, precision)[:, :nvs[precision]])
        Y = gpu_apply(hp, Xin, precision)
        want = P.apply(Xin) if precision == fk.FE_KS_F32 else ref[:, :nvs[precision]]
        assert parity_err(Y, want) <= TOL[precision], precision


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("p", [4, 6, 7, 8])
def test_more_points_than_nodes_and_scaled(p, cplx):
    wl = _wl(p, cplx, 0.05, nqx=2, n_v=9)
    hp, X = HostProblem(wl), trial_vectors(wl)
    P = Problem(wl)
    s = 1.0 / np.sqrt(P.lumped_mass())
    for precision in PREC:
        Xin = round_input(X, precision)
        ref = s[:, None] * P.apply(s[:, None] * Xin)
        for nv in (1, 8, 9):
            Y = gpu_apply(hp, np.ascontiguousarray(Xin[:, :nv]), precision, scaled=True)
            assert parity_err(Y, ref[:, :nv]) <= TOL[precision], (precision, nv)


@pytest.mark.parametrize("precision", PREC)
def test_same_bits_twice(precision):
    wl = dataclasses.replace(_wl(6, False, 0.05, n=3), n_v=21)
    hp, X = HostProblem(wl), round_input(trial_vectors(wl), precision)
    a, b = gpu_apply(hp, X, precision, repeat=2)
    assert np.array_equal(a, b)


TC = (fk.FE_KS_BF16, fk.FE_KS_F16, fk.FE_KS_BF16X2)


@pytest.mark.parametrize("precision,p,cplx,nv", [(q, 5, False, 13) for q in PREC] + [
    (q, p, cplx, nv) for q in TC for p in (3, 8) for cplx in (False, True) for nv in (13, 24)])
def test_one_launch_gives_the_bits_of_the_colour_launches(precision, p, cplx, nv):
    """Operator without projectors: the set-up stream takes the one-launch assembly, another
    stream and a captured graph go colour by colour; all the same bits."""
    wl = _wl(p, cplx, 0.05, n=3, n_atoms=0, n_v=nv)
    hp = HostProblem(wl)
    X = torch.from_numpy(trial_vectors(wl)).cuda().to(torch_dtype(precision, cplx))
    ys = [torch.full_like(X, float("nan")) for _ in range(3)]
    side = torch.cuda.Stream()
    home = torch.cuda.Stream()
    torch.cuda.synchronize()
    ctx = fk.fe_ks_setup(hp.struct, fk.TERM_ALL, wl.n_v, home.cuda_stream)
    try:
        fk.fe_ks_apply(ctx, X, ys[0], wl.n_v, precision)
        fk.fe_ks_set_stream(ctx, side.cuda_stream)
        fk.fe_ks_apply(ctx, X, ys[1], wl.n_v, precision)
        torch.cuda.synchronize()
        fk.fe_ks_set_stream(ctx, home.cuda_stream)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.stream(home):
            graph.capture_begin()
            fk.fe_ks_apply(ctx, X, ys[2], wl.n_v, precision)
            graph.capture_end()
        graph.replay()
        torch.cuda.synchronize()
    finally:
        fk.fe_ks_destroy(ctx)
    assert not torch.isnan(ys[0]).any()
    assert torch.equal(ys[0], ys[1]) and torch.equal(ys[0], ys[2])


@pytest.mark.parametrize("wide,narrow", [(fk.FE_KS_F64, fk.FE_KS_F32), (fk.FE_KS_F64E, fk.FE_KS_BF16)])
def test_storage_widths_of_one_context_overlap(wide, narrow):
    """An operator with projectors applied in FP64 and in FP32 storage on two streams, the FP32 ones
    as replays of a captured graph: the bits of applications one after the other."""
    wl = _wl(6, False, 0.05, n=4, n_v=40)
    hp = HostProblem(wl)
    X = torch.from_numpy(trial_vectors(wl)).cuda()
    X32 = X.float()
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    ctx = fk.fe_ks_setup(hp.struct, fk.TERM_ALL, wl.n_v, a.cuda_stream)
    try:
        ref, ref32 = torch.empty_like(X), torch.empty_like(X32)
        torch.cuda.synchronize()
        fk.fe_ks_apply(ctx, X, ref, wl.n_v, wide)
        fk.fe_ks_apply(ctx, X32, ref32, wl.n_v, narrow)
        torch.cuda.synchronize()
        y32 = torch.empty_like(X32)
        fk.fe_ks_set_stream(ctx, b.cuda_stream)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.stream(b):
            graph.capture_begin()
            for _ in range(4):
                fk.fe_ks_apply(ctx, X32, y32, wl.n_v, narrow)
            graph.capture_end()
        fk.fe_ks_set_stream(ctx, a.cuda_stream)
        ys = [torch.full_like(X, float("nan")) for _ in range(8)]
        for _ in range(5):
            y32.fill_(float("nan"))
            torch.cuda.synchronize()
            with torch.cuda.stream(b):
                graph.replay()
            for y in ys:
                fk.fe_ks_apply(ctx, X, y, wl.n_v, wide)
            torch.cuda.synchronize()
            assert torch.equal(y32, ref32)
            assert all(torch.equal(y, ref) for y in ys)
    finally:
        fk.fe_ks_destroy(ctx)


def _with_and_without_slots(hp, n_v, apply):
    """[apply(ctx)] of a context with assembly slots and of one without, on the same operator."""
    out = []
    try:
        for kind in (0, 1):
            fk.fe_ks_inject_setup_fault(kind)
            ctx = fk.fe_ks_setup(hp.struct, fk.TERM_ALL, n_v, torch.cuda.current_stream().cuda_stream)
            try:
                out.append(apply(ctx))
                torch.cuda.synchronize()
            finally:
                fk.fe_ks_destroy(ctx)
    finally:
        fk.fe_ks_inject_setup_fault(0)
    return out


FORMS = [(5, 3, 3), (5, 4, 72), (8, 3, 40), (8, 3, 41)]   # p, cells a side, columns: small tiles, wide x 3


@pytest.mark.parametrize("p,n,nv", FORMS)
@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("precision", PREC + list(TC))
def test_projectors_by_colour_and_in_one_launch(precision, cplx, p, n, nv):
    """Operator with projectors: the expansion reaches the slots and the scatter by colour with the same
    bits, in the small, flat and wide forms and in the tensor-core kernels, plain and scaled."""
    hp = HostProblem(_wl(p, cplx, 0.05, n=n, n_v=nv))
    X = torch.from_numpy(trial_vectors(_wl(p, cplx, 0.05, n=n, n_v=nv))).cuda().to(torch_dtype(precision, cplx))

    def apply(ctx):
        ys = [torch.full_like(X, float("nan")) for _ in range(2)]
        fk.fe_ks_apply(ctx, X, ys[0], nv, precision)
        fk.fe_ks_apply_scaled(ctx, X, ys[1], nv, precision)
        return ys

    one, colour = _with_and_without_slots(hp, nv, apply)
    assert not any(torch.isnan(y).any() for y in one)
    assert torch.equal(one[0], colour[0]) and torch.equal(one[1], colour[1])


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("precision", PREC + list(TC))
def test_filter_by_colour_and_in_one_launch(precision, cplx):
    """The filter's accumulating applications (Y += a H X) add to each row in the same order either way."""
    p, n, nv = 8, 3, 40
    wl = _wl(p, cplx, 0.05, n=n, n_v=nv)
    hp = HostProblem(wl)
    X = torch.from_numpy(trial_vectors(wl)).cuda()
    ritz = torch.linspace(0.0, 5.0, nv, dtype=torch.float64, device="cuda")

    def apply(ctx):
        nb = fk.fe_ks_cheb_filter_workspace(ctx, nv, precision)
        work = torch.empty(nb + 256, dtype=torch.uint8, device="cuda")
        work = work[(-work.data_ptr()) % 256:][:nb]
        y = X.clone()
        fk.fe_ks_cheb_filter(ctx, y, ritz, nv, 5, 0.0, 10.0, 4000.0, precision, work, nb)
        torch.cuda.synchronize()
        return y

    one, colour = _with_and_without_slots(hp, nv, apply)
    assert torch.isfinite(torch.view_as_real(one) if cplx else one).all()
    assert torch.equal(one, colour)


@pytest.mark.parametrize("p,nqx,cplx,first", [(1, 0, False, 500000), (2, 0, True, 300000), (3, 0, False, 280000),
                                              (1, 2, True, 280000), (4, 0, False, 160000), (2, 2, True, 160000),
                                              (5, 0, True, 60000), (3, 2, False, 60000), (7, 2, False, 25000)])
def test_large_blocks_in_pairs_of_floats(p, nqx, cplx, first):
    """Blocks on both sides of the line from which the pairs of floats take the kernel by tiles and
    colours: every column as a small block of the line kernel gives it, to rounding; the same bits twice
    and with and without slots; the block below the line in one launch."""
    n, cw = 4, 2 if cplx else 1
    nv = -(-first // (n ** 3 * cw))
    wl = _wl(p, cplx, 0.05, nqx=nqx, n=n, n_v=nv)
    hp = HostProblem(wl)
    X = torch.from_numpy(trial_vectors(wl)).cuda()
    some = torch.tensor([0, 1, 2, nv // 2, nv - 3, nv - 2], device="cuda")

    def apply(ctx):
        out = []
        for cols in (nv, nv, nv - 1, None):
            x = X[:, some].contiguous() if cols is None else X[:, :cols].contiguous()
            y = torch.full_like(x, float("nan"))
            fk.fe_ks_set_profiling(ctx, 1)
            fk.fe_ks_apply(ctx, x, y, x.shape[1], fk.FE_KS_F64E)
            out.append((y, fk.fe_ks_read_profile(ctx)["fill"][1]))
        return out

    one, colour = _with_and_without_slots(hp, nv, apply)
    (a, fa), (b, _), (below, fb), (small, _) = one
    assert torch.equal(a, b) and torch.equal(a, colour[0][0])
    assert (fa, fb) == (1, 0)                  # launches by colour start from a zero-fill, one launch does not
    small = small.cpu().numpy()
    for y in (a, below):
        assert not torch.isnan(y).any()
        assert parity_err(y[:, some].cpu().numpy(), small) <= TOL[fk.FE_KS_F64E]


def test_set_up_on_a_full_device_keeps_no_slots():
    """Set-up whose last slot allocation fails holds the memory of one without slots and gives the
    same bits; one with slots holds at least their size more."""
    wl = _wl(6, False, 0.05, n=6, n_v=64)
    hp = HostProblem(wl)
    X = torch.from_numpy(trial_vectors(wl)).cuda()
    stream = torch.cuda.current_stream().cuda_stream
    cells_per_dof = np.bincount(hp.dofs.ravel())
    slots = int(cells_per_dof[cells_per_dof > 1].sum()) * wl.n_v * (8 + 4)
    assert slots > 32 << 20
    granule = 4 << 20                      # small allocations share device pages
    try:
        for _ in range(5):                 # the first set-up may load modules; others may use the device
            ys, held = [], []
            for kind in (0, 1, 2):
                fk.fe_ks_inject_setup_fault(kind)
                torch.cuda.synchronize()
                free = torch.cuda.mem_get_info()[0]
                ctx = fk.fe_ks_setup(hp.struct, fk.TERM_ALL, wl.n_v, stream)
                try:
                    held.append(free - torch.cuda.mem_get_info()[0])
                    Y = torch.full_like(X, float("nan"))
                    fk.fe_ks_apply(ctx, X, Y, wl.n_v, fk.FE_KS_F64)
                    ys.append(Y)
                    torch.cuda.synchronize()
                finally:
                    fk.fe_ks_destroy(ctx)
            if abs(held[2] - held[1]) <= granule and held[0] - held[1] >= slots - granule:
                break
        else:
            raise AssertionError(f"held {held}, slots {slots}")
    finally:
        fk.fe_ks_inject_setup_fault(0)
    assert not torch.isnan(ys[0]).any() and all(torch.equal(ys[0], y) for y in ys)
    with pytest.raises(fk.FeKsError, match="ERR_ARG"):
        fk.fe_ks_inject_setup_fault(3)


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("precision", PREC)
def test_projection_column_groups(precision, cplx):
    """Column counts around the pair projection's splits of a block: 1, 3, 5, 12, 16, 33, 86, 129 and
    257 groups of 16 bytes, a column short of whole groups and not."""
    cols = 16 // (4 if precision == fk.FE_KS_F32 else 8) / (2 if cplx else 1)
    nvs = sorted({max(1, int(g * cols) - d) for g in (1, 3, 5, 12, 16, 33, 86, 129, 257) for d in (0, 1)})
    wl = _wl(2, cplx, 0.05, n=3, n_v=max(nvs))
    hp, X = HostProblem(wl), round_input(trial_vectors(wl), precision)
    ref = Problem(wl).apply(X)
    for nv in nvs:
        Y = gpu_apply(hp, np.ascontiguousarray(X[:, :nv]), precision)
        assert parity_err(Y, ref[:, :nv]) <= TOL[precision], nv
