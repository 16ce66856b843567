"""Performance cases of the finite-element Kohn-Sham operator library.

The listed cases are the calls an eigensolver program makes through the C
interface's Python binding: the operator application Y = H X in every
precision and operator type, the Chebyshev filter, the Rayleigh-Ritz step, the
Lanczos bound and the batched application of several small systems.  Meshes
are periodic n x n x n grids of hexahedra of degree p; fields, atoms and
trial blocks are seeded and evaluated here, and ``exact`` evaluates the same
operator in 64 bits with plain torch, from the definitions.
"""
import math

import numpy as np
import torch

from paper_2512_08571_gb300 import fe_ks as fk

H_CELL = 1.25            # bohr, cell size of the benchmark meshes
N_PROJ = 9               # l = 0, 1, 2 projectors of an atom
PROJ_L = [0, 1, 1, 1, 2, 2, 2, 2, 2]
PROJ_SIGMA, PROJ_RC = 0.8, 2.5
PREC = {"f64": fk.FE_KS_F64, "f32": fk.FE_KS_F32, "f64e": fk.FE_KS_F64E,
        "bf16": fk.FE_KS_BF16, "f16": fk.FE_KS_F16, "bf16x2": fk.FE_KS_BF16X2}
WIDE = ("f64", "f64e")   # stored in 64 bits; the others in 32


def _case(kind, p, n, nv, prec, name=None, nqx=0, cplx=False, jitter=0.0, gga=True, atoms=0, scaled=False,
          tuned=False, degree=0, steps=0, systems=0):
    c = dict(kind=kind, p=p, n=n, nv=nv, prec=prec, nqx=nqx, cplx=cplx, jitter=jitter, gga=gga, atoms=atoms,
             scaled=scaled, tuned=tuned, degree=degree, steps=steps, systems=systems)
    if name is not None:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest problem of the benchmark (4^3 cells, p = 4, 8 vectors, T + V_loc): launches and latency
        _case("apply", 4, 4, 8, "f64", "apply_f64_small", gga=False),
        # the jittered pseudopotential mesh in native FP64, D^{-1/2} H D^{-1/2} as the eigensolver applies it
        _case("apply", 6, 10, 64, "f64", "apply_f64_jitter", jitter=0.1, atoms=9, scaled=True),
        # FP32 with a block size that is no multiple of a vector load (a locked, shrunken block)
        _case("apply", 6, 12, 37, "f32", "apply_f32_ragged", jitter=0.1, atoms=16),
        # a Bloch (complex) operator at one k point
        _case("apply", 7, 10, 64, "f32", "apply_f32_bloch", cplx=True, atoms=8),
        # the paper's default quadrature n_q = n_p + 2
        _case("apply", 8, 8, 32, "f32", "apply_f32_nq2", nqx=2, atoms=3),
        # the headline shape in FP32 (p = 8, 256 vectors), tuned as a long-running program tunes it; the largest
        _case("apply", 8, 16, 256, "f32", "apply_f32_headline", atoms=19, tuned=True),
        # the same shape with BF16 tensor-core contractions, on a smaller mesh
        _case("apply", 8, 12, 256, "bf16", "apply_bf16_headline", atoms=8),
        # the FP64-accurate application on the FP32 pipe: residuals and Rayleigh-Ritz
        _case("apply", 8, 8, 64, "f64e", "apply_f64e", atoms=3, scaled=True),
        # one Chebyshev filter of the eigensolver: FP32 recurrence, FP64-accurate residual
        _case("filter", 6, 8, 48, "f32", "filter_mixed", atoms=5, degree=20),
        # one Rayleigh-Ritz step of the eigensolver (FP64-accurate plan)
        _case("rr", 6, 10, 96, "f64e", "rayleigh_ritz", atoms=9),
        # the spectral bound that precedes the filter: ten applications to one vector
        _case("lanczos", 8, 12, 1, "f64e", "lanczos_bound", atoms=8, steps=10),
        # several small systems in one call (k points, images, screening runs)
        _case("batch", 4, 4, 8, "f64", "batch_small", systems=8),
    ]


def _rel_cost(case):
    """Rough relative time of a pass, for keeping drawn cases within the largest listed one."""
    rate = {"f64": 1 / 25, "f64e": 1 / 8, "f32": 1.0, "bf16": 1.0, "f16": 1.0, "bf16x2": 1 / 2.8}[case["prec"]]
    if case["kind"] == "lanczos":
        return 16 * work(case)["flops"] / rate
    return work(case)["flops"] / rate


def draw(rng):
    limit = max(_rel_cost(c) for c in listed())

    def logi(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    while True:
        kind = rng.choice(["apply"] * 8 + ["filter", "filter", "rr", "lanczos", "batch"])
        p, n, nv = rng.randint(3, 8), logi(3, 16), logi(1, 256)
        jitter = rng.choice([0.0, 0.1])
        if kind == "apply":
            prec = rng.choice(["f32", "f32", "f32", "f64", "f64", "f64e", "bf16", "f16", "bf16x2"])
            nqx = 2 if prec in ("f32", "f64", "f64e") and rng.random() < 0.2 else 0
            c = _case("apply", p, n, nv, prec, nqx=nqx, cplx=rng.random() < 0.3, jitter=jitter,
                      gga=rng.random() < 0.8, atoms=rng.choice([0, max(1, n ** 3 // 200)]),
                      scaled=rng.random() < 0.4, tuned=rng.random() < 0.25)
        elif kind == "filter":
            c = _case("filter", p, n, nv, rng.choice(["f32", "f32", "bf16", "f64e"]), cplx=rng.random() < 0.2,
                      jitter=jitter, atoms=rng.choice([0, max(1, n ** 3 // 200)]), degree=rng.randint(8, 24))
        elif kind == "rr":
            c = _case("rr", p, max(4, n), min(160, max(4, nv)), "f64e", jitter=jitter, atoms=max(1, n ** 3 // 200))
        elif kind == "lanczos":
            c = _case("lanczos", p, n, 1, rng.choice(["f64", "f64e"]), cplx=rng.random() < 0.3, jitter=jitter,
                      atoms=max(1, n ** 3 // 200), steps=rng.randint(8, 14))
        else:
            c = _case("batch", rng.randint(4, 6), rng.randint(3, 5), rng.randint(4, 16), "f64",
                      systems=rng.randint(4, 12))
        # a Rayleigh-Ritz block stays far from filling the space
        if _rel_cost(c) <= limit and (c["kind"] != "rr" or (n * p) ** 3 >= 16 * c["nv"]):
            return c


# ------------------------------------------------------------------ inputs

def _systems(case):
    """The systems of a batch case: uneven grids, degrees, block sizes; FP64 and FP32 in turn."""
    out = []
    for s in range(case["systems"]):
        out.append(_case("apply", 4 + (case["p"] + s) % 5, case["n"] + s % 3, case["nv"] * (1 + s % 4),
                         "f64" if s % 2 == 0 else "f32", atoms=1 + s % 3))
    return out


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 7919 + 17)
    return g


class _Problem:
    """Mesh, fields, atoms and projector values of one system, evaluated at the library's quadrature points."""

    def __init__(self, case, seed):
        rng = np.random.default_rng(int(seed) * 1009 + 11)
        n, p = case["n"], case["p"]
        self.case, self.n, self.p, self.nq = case, n, p, p + 1 + case["nqx"]
        self.L = L = H_CELL * n
        c = np.arange(n)
        cz, cy, cx = (a.ravel() for a in np.meshgrid(c, c, c, indexing="ij"))
        move = rng.uniform(-1.0, 1.0, (n, n, n, 3)) * case["jitter"] * H_CELL
        self.verts = np.empty((n ** 3, 8, 3))
        for v in range(8):
            gx, gy, gz = cx + (v & 1), cy + ((v >> 1) & 1), cz + ((v >> 2) & 1)
            self.verts[:, v] = np.stack([gx, gy, gz], axis=1) * H_CELL + move[gz % n, gy % n, gx % n]
        M = n * p
        li = np.arange(p + 1)
        k, j, i = (a.ravel() for a in np.meshgrid(li, li, li, indexing="ij"))
        self.dofs = np.ascontiguousarray((cx[:, None] * p + i) % M + M * ((cy[:, None] * p + j) % M +
                                         M * ((cz[:, None] * p + k) % M)), dtype=np.int32)
        self.m = M ** 3
        self.kpt = np.array([0.25, 0.1, 0.15]) * 2 * math.pi / L if case["cplx"] else np.zeros(3)
        s = self.struct = fk.fe_ks_problem()
        s.n_cells, s.n_dofs, s.degree, s.n_q = n ** 3, self.m, p, self.nq
        s.cell_vertices, s.cell_dofs = self.verts.ctypes.data, self.dofs.ctypes.data
        xq = torch.from_numpy(fk.fe_ks_quadrature_points(s)).cuda()
        # V_loc: four periodic Gaussian wells; V^G: three periodic sine waves
        vl = torch.zeros(xq.shape[:2], dtype=torch.float64, device="cuda")
        for _ in range(4):
            a, w, c0 = rng.uniform(1.0, 5.0), rng.uniform(0.5, 1.5), rng.uniform(0.0, L, 3)
            prod = torch.full_like(vl, -a)
            for ax in range(3):
                d = xq[..., ax] - c0[ax]
                prod *= sum(torch.exp(-(d - sh * L) ** 2 / (2 * w * w)) for sh in (-1, 0, 1))
            vl += prod
        self.vloc = vl.cpu().numpy()
        self.vgga = None
        waves = [(rng.uniform(-0.5, 0.5, 3), rng.integers(0, 2, 3), rng.uniform(0, 2 * math.pi)) for _ in range(3)]
        if case["gga"]:
            vg = torch.zeros_like(xq)
            for a, nj, ph in waves:
                arg = 2 * math.pi / L * (xq @ torch.tensor(nj, dtype=torch.float64, device="cuda")) + ph
                vg += torch.sin(arg)[..., None] * torch.tensor(a, device="cuda")
            self.vgga = vg.cpu().numpy()
            s.v_gga_q = self.vgga.ctypes.data
        s.v_loc_q = self.vloc.ctypes.data
        for d in range(3):
            s.kpt[d] = float(self.kpt[d])
        s.force_complex = int(case["cplx"])
        s.n_atoms, s.n_proj = 0, N_PROJ
        if case["atoms"]:
            self._atoms(rng, xq)

    def _atoms(self, rng, xq):
        s, L, A = self.struct, self.L, self.case["atoms"]
        R = rng.uniform(0.0, L, (A, 3))
        self.h = np.ascontiguousarray(rng.uniform(-2.0, 2.0, (A, 3))[:, PROJ_L])
        cen = self.verts.mean(axis=1)
        rad = np.linalg.norm(self.verts - cen[:, None], axis=-1).max(axis=1)
        g = np.array([-L, 0.0, L])
        img = np.stack(np.meshgrid(g, g, g, indexing="ij"), axis=-1).reshape(-1, 3)
        ptr, cells, shifts = [0], [], []
        for a in range(A):
            dist = np.linalg.norm(cen[:, None] - (R[a] + img)[None], axis=-1)
            ce, im = np.nonzero(dist < PROJ_RC + rad[:, None])
            cells.append(ce)
            shifts.append(img[im])
            ptr.append(ptr[-1] + len(ce))
        self.ptr = np.array(ptr, dtype=np.int32)
        self.cells = np.concatenate(cells).astype(np.int32)
        self.shift = np.ascontiguousarray(np.concatenate(shifts))
        at = np.repeat(np.arange(A), np.diff(self.ptr))
        d = xq[torch.from_numpy(self.cells).long().cuda()] - torch.from_numpy(R[at] + self.shift).cuda()[:, None]
        x, y, z = d.unbind(-1)
        r2 = x * x + y * y + z * z
        rad = torch.exp(-r2 / (2 * PROJ_SIGMA ** 2)) * (1 - r2 / PROJ_RC ** 2).clamp(min=0) ** 3
        c1, c2, c0 = math.sqrt(3 / (4 * math.pi)), math.sqrt(15 / math.pi), math.sqrt(5 / math.pi)
        ylm = [torch.full_like(x, 0.5 / math.sqrt(math.pi)), c1 * y, c1 * z, c1 * x, 0.5 * c2 * x * y, 0.5 * c2 * y * z,
               0.25 * c0 * (3 * z * z - r2), 0.5 * c2 * x * z, 0.25 * c2 * (x * x - y * y)]
        self.chi = (rad[..., None] * torch.stack(ylm, dim=-1)).contiguous().cpu().numpy()
        s.n_atoms = A
        s.atom_cell_ptr, s.atom_cells = self.ptr.ctypes.data, self.cells.ctypes.data
        s.image_shift, s.chi_q, s.h_coef = self.shift.ctypes.data, self.chi.ctypes.data, self.h.ctypes.data

    def waves(self, nv):
        """The nv longest periodic plane waves (real: cosines and sines), by kinetic energy: [(G, phase)]."""
        top = 1
        while (2 * top + 1) ** 3 < 2 * nv + 2:
            top += 1
        ks = np.array([(a, b, c) for a in range(-top, top + 1) for b in range(-top, top + 1) for c in range(-top, top + 1)])
        ks = ks[np.argsort((ks ** 2).sum(axis=1), kind="stable")]
        if self.case["cplx"]:
            return [(2 * math.pi / self.L * k, 0.0) for k in ks[:nv]]
        half = [k for k in ks if tuple(k) >= (0, 0, 0)]
        both = [(2 * math.pi / self.L * k, ph) for k in half for ph in (0.0, -0.5 * math.pi) if k.any() or ph == 0.0]
        return both[:nv]

    def bounds(self, nv):
        """(lam_min, lam_T, lam_max) for the filter of nv plane waves: below the wells, the end of the wanted
        part, and an upper bound of the largest eigenvalue of one cell's kinetic operator."""
        x, w, xn, wn, N, dN = _tables(self.p, self.p + 1)
        K = (dN * w[:, None]).T @ dN * 2 / H_CELL
        s = 1 / np.sqrt(wn * H_CELL / 2)
        top = 1.5 * np.linalg.eigvalsh(s[:, None] * K * s[None])[-1]
        top = top * (1.6 if self.case["jitter"] else 1.0) + 60.0
        return -5.0, float(self.energies(nv)[-1]) + 1.0, top

    def energies(self, nv):
        e = np.array([0.5 * float((G + self.kpt) @ (G + self.kpt)) for G, _ in self.waves(nv)])
        return np.sort(e) - 1.0 + 1e-3 * np.arange(nv)


class _State:
    """What a program holds between calls; frees the library's handles with itself."""

    def __init__(self, case):
        self.case, self.ctxs, self.batch = case, [], None

    def __del__(self):
        if self.batch is not None:
            fk.fe_ks_batch_destroy(self.batch)
        for c in self.ctxs:
            fk.fe_ks_destroy(c)

    def setup(self, problem, nv):
        ctx = fk.fe_ks_setup(problem.struct, fk.TERM_ALL, nv, torch.cuda.current_stream().cuda_stream)
        self.ctxs.append(ctx)
        return ctx


def _block(problem, nv, prec, g):
    """A trial block, uniform in [-1, 1], in the precision's storage type."""
    shape = (problem.m, nv) + ((2,) if problem.case["cplx"] else ())
    x = torch.empty(shape, dtype=torch.float64 if prec in WIDE else torch.float32, device="cuda")
    x.uniform_(-1.0, 1.0, generator=g)
    return torch.view_as_complex(x) if problem.case["cplx"] else x


def _aligned(nbytes):
    buf = torch.empty(nbytes + 256, dtype=torch.uint8, device="cuda")
    off = (-buf.data_ptr()) % 256
    return buf[off:off + nbytes]


def prepare(case, seed):
    st = _State(case)
    kind, nv, prec = case["kind"], case["nv"], case["prec"]
    g = _gen(seed)
    if kind == "batch":
        st.X, st.Y, systems = [], [], _systems(case)
        for i, c in enumerate(systems):
            pr = _Problem(c, seed * 64 + i)
            st.setup(pr, c["nv"])
            st.X.append(_block(pr, c["nv"], c["prec"], g))
            st.Y.append(torch.empty_like(st.X[-1]))
        st.batch = fk.fe_ks_batch_create(st.ctxs, [c["nv"] for c in systems], [PREC[c["prec"]] for c in systems])
        return st
    pr = _Problem(case, seed)
    ctx = st.setup(pr, nv)
    if kind == "apply":
        st.X = _block(pr, nv, prec, g)
        st.Y = torch.empty_like(st.X)
        if case["tuned"]:
            fk.fe_ks_tune(ctx, st.X, st.Y, nv, PREC[prec], reps=1)
    elif kind == "lanczos":
        st.nbytes = fk.fe_ks_lanczos_bound_workspace(ctx, case["steps"])
        st.work = _aligned(st.nbytes)
        st.v0 = _start_vector(pr, g)
    elif kind == "filter":
        st.nbytes = fk.fe_ks_cheb_filter_workspace(ctx, nv, PREC[prec])
        st.work = _aligned(st.nbytes)
        st.X0 = _ritz_like(pr, nv, g)
        st.X = torch.empty_like(st.X0)
        st.bounds = pr.bounds(nv)
        st.ritz = torch.from_numpy(pr.energies(nv)).cuda()
    else:
        st.nbytes = fk.fe_ks_rayleigh_ritz_workspace(ctx, nv, PREC[prec])
        st.work = _aligned(st.nbytes)
        st.X0 = _ritz_like(pr, nv, g)
        st.X = torch.empty_like(st.X0)
        st.ritz = torch.empty(nv, dtype=torch.float64, device="cuda")
    return st


def _start_vector(problem, g):
    v = torch.empty((problem.m, 1) + ((2,) if problem.case["cplx"] else ()), dtype=torch.float64, device="cuda")
    v.normal_(generator=g)
    return torch.view_as_complex(v) if problem.case["cplx"] else v


def _ritz_like(problem, nv, g):
    """A block as the previous pass leaves it: D^{1/2} times smooth functions (the longest plane waves) and a few
    percent of everything else, columns of about unit norm."""
    x, w, xn, wn, N, dN = _tables(problem.p, problem.nq)
    Z, Y, X = (t.ravel() for t in np.meshgrid(xn, xn, xn, indexing="ij"))
    pos = np.empty((problem.m, 3))
    pos[problem.dofs.ravel()] = _points(problem.verts, X, Y, Z).reshape(-1, 3)
    D = torch.zeros(problem.m, dtype=torch.float64, device="cuda")
    D.index_add_(0, torch.from_numpy(problem.dofs).cuda().long().ravel(), _geometry(problem.verts, xn, wn)[1].ravel())
    G, ph = zip(*problem.waves(nv))
    arg = torch.from_numpy(pos).cuda() @ torch.from_numpy(np.array(G)).cuda().T + torch.tensor(ph, device="cuda", dtype=torch.float64)
    wave = torch.polar(torch.ones_like(arg), arg) if problem.case["cplx"] else torch.cos(arg)
    wave *= D.sqrt()[:, None]
    wave /= torch.linalg.vector_norm(wave, dim=0)
    return (wave + 0.03 * math.sqrt(3.0 / problem.m) * _block(problem, nv, "f64", g)).contiguous()


def _points(verts, X, Y, Z):
    """Physical positions [cell][point][3] of the reference points (X, Y, Z)."""
    out = 0.0
    for v in range(8):
        f = (1 + (2 * (v & 1) - 1) * X) * (1 + (2 * ((v >> 1) & 1) - 1) * Y) * (1 + (2 * ((v >> 2) & 1) - 1) * Z) / 8
        out = out + f[None, :, None] * verts[:, None, v]
    return out


# ------------------------------------------------------------------ one pass

def run(state):
    case = state.case
    kind, nv, prec = case["kind"], case["nv"], PREC[case["prec"]]
    if kind == "batch":
        fk.fe_ks_batch_apply(state.batch, state.X, state.Y, torch.cuda.current_stream().cuda_stream)
        return state.Y
    ctx = state.ctxs[0]
    if kind == "apply":
        (fk.fe_ks_apply_scaled if case["scaled"] else fk.fe_ks_apply)(ctx, state.X, state.Y, nv, prec)
        return state.Y
    if kind == "lanczos":
        top, alpha, beta = fk.fe_ks_lanczos_bound(ctx, state.v0, case["steps"], prec, state.work, state.nbytes)
        return {"lam_max": top, "alpha": np.array(alpha), "beta": np.array(beta)}
    state.X.copy_(state.X0)      # the outer loop hands every pass a new block; both steps work in place
    if kind == "filter":
        fk.fe_ks_cheb_filter(ctx, state.X, state.ritz, nv, case["degree"], *state.bounds, prec, state.work,
                             state.nbytes, residual_precision=fk.FE_KS_F64E)
        return state.X
    fk.fe_ks_rayleigh_ritz(ctx, state.X, state.ritz, nv, prec, state.work, state.nbytes)
    return {"ritz": state.ritz, "X": state.X}


# ------------------------------------------------------------------ work and tolerance

def _line(a, b):
    """Flops of one 1D contraction a -> b with the even-odd split."""
    return a + a * b + b


def _apply_work(case):
    p, n = case["p"], case["n"]
    a, q = p + 1, p + 1 + case["nqx"]
    E, cw = n ** 3, 2 if case["cplx"] else 1
    cols, size = case["nv"] * cw, 8 if case["prec"] in WIDE else 4
    flops = 2 * (a * a * _line(a, q) + a * q * _line(a, q) + q * q * _line(a, q)) + 6 * q * q * _line(q, q)
    flops += q ** 3 * (16 + (12 if case["gga"] else 0) + (6 if case["cplx"] else 0))
    ncoef = 7 + (3 if case["gga"] else 0) + (3 if case["cplx"] else 0)
    pairs = 100 * case["atoms"]       # about a hundred cells meet an atom's support at h = 1.25
    flops = E * cols * flops + 4 * pairs * N_PROJ * a ** 3 * cols * cw
    nbytes = E * (ncoef * q ** 3 * size + 4 * a ** 3) + pairs * N_PROJ * a ** 3 * size * cw
    return float(flops), float(nbytes), 2.0 * (n * p) ** 3 * cols * size


def work(case):
    if case["kind"] == "batch":
        parts = [work(c) for c in _systems(case)]
        return {k: sum(w[k] for w in parts) for k in ("bytes", "flops")}
    flops, tables, xy = _apply_work(case)
    m = (case["n"] * case["p"]) ** 3
    if case["kind"] == "apply":
        return {"bytes": tables + xy, "flops": flops}
    if case["kind"] == "lanczos":
        return {"bytes": case["steps"] * (tables + xy), "flops": case["steps"] * flops}
    wide = 2.0 * m * case["nv"] * (2 if case["cplx"] else 1) * 8
    if case["kind"] == "filter":      # every step reads and writes the recurrence's blocks
        return {"bytes": case["degree"] * (tables + 2 * xy) + 2 * wide, "flops": case["degree"] * flops}
    return {"bytes": tables + xy + 3 * wide, "flops": flops + 6.0 * m * case["nv"] ** 2}


def tolerance(case):
    """About four times the difference from ``exact`` (see there), by the arithmetic of the call."""
    kind, prec = case["kind"], case["prec"]
    if kind == "rr":
        return {"rel": 1e-10}         # eigenvectors of Ritz values a small gap apart
    if kind == "lanczos":
        return {"rel": 1e-12}
    if kind == "batch":
        return {"rel": 1e-6}
    if kind == "filter":
        return {"rel": {"f32": 1e-5, "bf16": 2e-2, "f64e": 2e-13}[prec]}
    return {"rel": {"f64": 2e-14, "f64e": 5e-14, "f32": 1e-6, "bf16": 1.3e-2, "f16": 2.2e-3, "bf16x2": 3e-5}[prec]}


# ------------------------------------------------------------------ the same in 64 bits

def _tables(p, nq):
    """Gauss points and weights, GLL nodes and weights, basis values N and derivatives dN at the Gauss points."""
    x, w = np.polynomial.legendre.leggauss(nq)
    leg = np.polynomial.legendre.Legendre.basis(p)
    inner = np.sort(np.real(leg.deriv().roots()))
    for _ in range(3):                # polish the roots of P_p'
        inner -= leg.deriv()(inner) / leg.deriv(2)(inner) if inner.size else 0.0
    xn = np.concatenate([[-1.0], inner, [1.0]])
    wn = 2.0 / (p * (p + 1) * leg(xn) ** 2)
    N, dN = np.ones((nq, p + 1)), np.zeros((nq, p + 1))
    for i in range(p + 1):
        for j in range(p + 1):
            if j != i:
                N[:, i] *= (x - xn[j]) / (xn[i] - xn[j])
        for k in range(p + 1):
            if k != i:
                t = np.full(nq, 1.0 / (xn[i] - xn[k]))
                for j in range(p + 1):
                    if j not in (i, k):
                        t *= (x - xn[j]) / (xn[i] - xn[j])
                dN[:, i] += t
    return x, w, xn, wn, N, dN


def _geometry(verts, x, w):
    """Inverse Jacobians and det J w of trilinear cells at the tensor points of x, index z, y, x."""
    q = len(x)
    Z, Y, X = (a.ravel() for a in np.meshgrid(x, x, x, indexing="ij"))
    W = (w[:, None, None] * w[None, :, None] * w[None, None, :]).ravel()
    d = np.zeros((8, 3, q ** 3))
    for v in range(8):
        s = [2 * (v & 1) - 1, 2 * ((v >> 1) & 1) - 1, 2 * ((v >> 2) & 1) - 1]
        f = [(1 + s[0] * X) / 2, (1 + s[1] * Y) / 2, (1 + s[2] * Z) / 2]
        for a in range(3):
            d[v, a] = s[a] / 2 * f[(a + 1) % 3] * f[(a + 2) % 3]
    J = torch.einsum("evc,vdq->eqcd", torch.from_numpy(verts).cuda(), torch.from_numpy(d).cuda())
    return torch.linalg.inv(J), torch.linalg.det(J) * torch.from_numpy(W).cuda()


def _contract(mats, u):
    """u[e, z, y, x, v] with a matrix along each axis (z, y, x)."""
    u = torch.einsum("qk,ekjiv->eqjiv", mats[0], u)
    u = torch.einsum("qj,ekjiv->ekqiv", mats[1], u)
    return torch.einsum("qi,ekjiv->ekjqv", mats[2], u)


class _Exact:
    """H X (scaled: D^{-1/2} H D^{-1/2} X) by quadrature over blocks of cells, in 64 bits."""

    def __init__(self, problem, scaled):
        self.P, self.scaled = problem, scaled
        x, w, xn, wn, N, dN = _tables(problem.p, problem.nq)
        self.dt = torch.complex128 if problem.case["cplx"] else torch.float64
        self.N, self.D = (torch.from_numpy(a).cuda().to(self.dt) for a in (N, dN))
        self.x, self.w = x, w
        self.dofs = torch.from_numpy(problem.dofs).cuda().long()
        D = torch.zeros(problem.m, dtype=torch.float64, device="cuda")
        D.index_add_(0, self.dofs.ravel(), _geometry(problem.verts, xn, wn)[1].ravel())
        self.s = D.rsqrt()[:, None]
        self.F = self._projectors() if problem.case["atoms"] else None

    def _projectors(self):
        P, a = self.P, self.P.p + 1
        cells = torch.from_numpy(P.cells).long()
        out = []
        for b in range(0, len(cells), 256):
            ce = cells[b:b + 256]
            wd = _geometry(P.verts[ce.numpy()], self.x, self.w)[1]
            chi = torch.from_numpy(P.chi[b:b + 256]).cuda().to(self.dt) * wd[..., None]
            if P.case["cplx"]:
                Z, Y, X = (t.ravel() for t in np.meshgrid(self.x, self.x, self.x, indexing="ij"))
                ph = (_points(P.verts[ce.numpy()], X, Y, Z) - P.shift[b:b + 256, None]) @ P.kpt
                chi = chi * torch.exp(-1j * torch.from_numpy(ph).cuda())[..., None]
            q = P.nq
            out.append(_contract([self.N.T] * 3, chi.reshape(len(ce), q, q, q, N_PROJ)).reshape(len(ce), a ** 3, N_PROJ))
        return torch.cat(out)

    def __call__(self, X):
        P, a, q = self.P, self.P.p + 1, self.P.nq
        X = X.to(self.dt)
        if self.scaled:
            X = X * self.s
        Y = torch.zeros_like(X)
        kpt = torch.from_numpy(P.kpt).cuda()
        block = max(1, 40_000_000 // (q ** 3 * X.shape[1] * (2 if P.case["cplx"] else 1)))
        for b in range(0, P.n ** 3, block):
            d = self.dofs[b:b + block]
            u = X[d].reshape(len(d), a, a, a, -1)
            Ji, wd = _geometry(P.verts[b:b + block], self.x, self.w)
            val = _contract([self.N] * 3, u).reshape(len(d), q ** 3, -1)
            ref = [_contract([self.D if ax == 2 - s else self.N for ax in range(3)], u).reshape(len(d), q ** 3, -1)
                   for s in range(3)]
            grad = [sum(Ji[..., s, c, None] * ref[s] for s in range(3)) for c in range(3)]
            vl = torch.from_numpy(P.vloc[b:b + block]).cuda() + 0.5 * float(P.kpt @ P.kpt)
            z = vl[..., None] * val
            flux = [0.5 * g for g in grad]
            if P.vgga is not None:
                vg = torch.from_numpy(P.vgga[b:b + block]).cuda()
                for c in range(3):
                    z = z + vg[..., c, None] * grad[c]
                    flux[c] = flux[c] + vg[..., c, None] * val
            if P.case["cplx"]:
                z = z - 1j * sum(kpt[c] * grad[c] for c in range(3))
            z = z * wd[..., None]
            flux = [f * wd[..., None] for f in flux]
            out = _contract([self.N.T] * 3, z.reshape(len(d), q, q, q, -1))
            for s in range(3):
                f = sum(Ji[..., s, c, None] * flux[c] for c in range(3)).reshape(len(d), q, q, q, -1)
                out = out + _contract([(self.D if ax == 2 - s else self.N).T for ax in range(3)], f)
            Y.index_add_(0, d.ravel(), out.reshape(d.numel(), -1))
        if self.F is not None:
            ce = torch.from_numpy(P.cells).long().cuda()
            at = torch.repeat_interleave(torch.arange(P.case["atoms"], device="cuda"),
                                         torch.from_numpy(np.diff(P.ptr)).long().cuda())
            Q = torch.zeros((P.case["atoms"], N_PROJ, X.shape[1]), dtype=self.dt, device="cuda")
            for b in range(0, len(ce), 256):
                Q.index_add_(0, at[b:b + 256], torch.einsum("pnb,pnv->pbv", self.F[b:b + 256].conj(),
                                                            X[self.dofs[ce[b:b + 256]]]))
            Q = Q * torch.from_numpy(P.h).cuda()[..., None]
            for b in range(0, len(ce), 256):
                d = self.dofs[ce[b:b + 256]]
                Y.index_add_(0, d.ravel(), torch.einsum("pnb,pbv->pnv", self.F[b:b + 256], Q[at[b:b + 256]])
                             .reshape(d.numel(), -1))
        return Y * self.s if self.scaled else Y


def exact(case, seed):
    """What ``run`` computes, from the definitions in 64 bits: the operator by quadrature, the filter as its
    Chebyshev polynomial, Rayleigh-Ritz by a dense eigensolve (the sign of a Ritz vector is free: no value),
    Lanczos by its recurrence."""
    kind, nv, g = case["kind"], case["nv"], _gen(seed)
    if kind == "batch":
        out = []
        for i, c in enumerate(_systems(case)):
            pr = _Problem(c, seed * 64 + i)
            out.append(_Exact(pr, False)(_block(pr, c["nv"], c["prec"], g)))
        return out
    pr = _Problem(case, seed)
    if kind == "apply":
        return _Exact(pr, case["scaled"])(_block(pr, nv, case["prec"], g))
    H = _Exact(pr, True)
    if kind == "lanczos":
        v = _start_vector(pr, g)
        v, prev, alpha, beta = v / torch.linalg.vector_norm(v), torch.zeros_like(v), [], []
        for _ in range(case["steps"]):
            w = H(v)
            alpha.append(torch.vdot(v.ravel(), w.ravel()).real.item())
            w = w - alpha[-1] * v - (beta[-1] if beta else 0.0) * prev
            beta.append(torch.linalg.vector_norm(w).item())
            prev, v = v, w / beta[-1]
        T = np.diag(alpha) + np.diag(beta[:-1], 1) + np.diag(beta[:-1], -1)
        return {"lam_max": float(np.linalg.eigvalsh(T)[-1] + beta[-1]), "alpha": np.array(alpha),
                "beta": np.array(beta)}
    X = _ritz_like(pr, nv, g)
    if kind == "filter":
        lmin, lt, top = pr.bounds(nv)
        e, c = 0.5 * (top - lt), 0.5 * (top + lt)
        s1 = s = e / (lmin - c)
        Y = (H(X) - c * X) * (s1 / e)
        for _ in range(2, case["degree"] + 1):
            s2 = 1 / (2 / s1 - s)
            X, Y, s = Y, (H(Y) - c * Y) * (2 * s2 / e) - (s * s2) * X, s2
        return Y
    L = torch.linalg.cholesky(X.T @ X)
    A = torch.linalg.solve_triangular(L, torch.linalg.solve_triangular(L, X.T @ H(X), upper=False).T, upper=False)
    return {"ritz": torch.linalg.eigvalsh(0.5 * (A + A.T)), "X": None}
