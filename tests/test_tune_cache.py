"""The tile-configuration cache: a context of the same shape picks up another
context's tuned configuration at its next application, unless its own was
set explicitly; the choice never changes the result beyond rounding."""
import numpy as np
import pytest

from paper_2512_08571_gb300 import fe_ks as fk
from synth.host_problem import HostProblem
from synth import CONFIGS, Workload, trial_vectors

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_tuned_configuration_is_shared_by_same_shape_contexts():
    wl = CONFIGS["C4"].scaled(n=4, n_v=16, n_atoms=3)
    hp = HostProblem(wl)
    st = torch.cuda.current_stream().cuda_stream
    X = torch.from_numpy(trial_vectors(wl).astype(np.float32)).cuda()
    Y = torch.empty_like(X)
    a = fk.fe_ks_setup(hp.struct, fk.TERM_ALL, wl.n_v, st)
    b = fk.fe_ks_setup(hp.struct, fk.TERM_ALL, wl.n_v, st)
    c = fk.fe_ks_setup(hp.struct, fk.TERM_ALL, wl.n_v, st)
    try:
        fk.fe_ks_set_config(c, fk.FE_KS_F32, 2)                 # explicit: keeps its own
        best, ms = fk.fe_ks_tune(a, X, Y, wl.n_v, fk.FE_KS_F32, reps=1)
        assert fk.fe_ks_get_config(a, fk.FE_KS_F32) == best
        assert fk.fe_ks_get_config(b, fk.FE_KS_F32) == 0        # not applied yet
        fk.fe_ks_apply(b, X, Y, wl.n_v, fk.FE_KS_F32)
        assert fk.fe_ks_get_config(b, fk.FE_KS_F32) == best
        Yc = torch.empty_like(X)
        fk.fe_ks_apply(c, X, Yc, wl.n_v, fk.FE_KS_F32)
        assert fk.fe_ks_get_config(c, fk.FE_KS_F32) == 2
        torch.cuda.synchronize()
        d = (Y - Yc).norm(dim=0) / Yc.norm(dim=0)
        assert float(d.max()) < 1e-5
    finally:
        for ctx in (a, b, c):
            fk.fe_ks_destroy(ctx)


def test_tuned_configuration_stays_with_its_size_and_assembly():
    """A choice made by colour (a context without assembly slots, where the pairs of floats at p = 6 prefer
    another configuration than the default) reaches a context of the same mesh without slots, and none
    with slots or with an eighth of the cells, whose default takes another form."""
    p, n_v, prec = 6, 64, fk.FE_KS_F64E
    big, small = (Workload("t", L=2.0 * n, n=n, p=p, nq=p + 1, n_v=n_v, gga=True, n_atoms=2, jitter=0.05, seed=99)
                  for n in (8, 4))
    hb, hs = HostProblem(big), HostProblem(small)
    st = torch.cuda.current_stream().cuda_stream
    X, Xs = torch.from_numpy(trial_vectors(big)).cuda(), torch.from_numpy(trial_vectors(small)).cuda()
    ctxs = []

    def setup(hp, kind):
        fk.fe_ks_inject_setup_fault(kind)
        try:
            ctxs.append(fk.fe_ks_setup(hp.struct, fk.TERM_ALL, n_v, st))
        finally:
            fk.fe_ks_inject_setup_fault(0)
        return ctxs[-1]

    try:
        best, ms = fk.fe_ks_tune(setup(hb, 1), X, torch.empty_like(X), n_v, prec, reps=5)
        if best == 0:
            pytest.skip("the tuner took the default")
        for hp, kind, x, want in ((hb, 1, X, best), (hb, 0, X, 0), (hs, 1, Xs, 0)):
            ctx = setup(hp, kind)
            fk.fe_ks_apply(ctx, x, torch.empty_like(x), n_v, prec)
            assert fk.fe_ks_get_config(ctx, prec) == want, (kind, x.shape)
        torch.cuda.synchronize()
    finally:
        for ctx in ctxs:
            fk.fe_ks_destroy(ctx)
