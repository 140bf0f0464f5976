"""What the sliced product has to take as the walks do: general contractions
with many functions per primitive, densities that are not finite, and very small
and very large ones; and what a caller sees of a bounded wait that gave up."""
import numpy as np
import pytest

from paper_2509_16460_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def F():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2509_16460_gb300 import build
    build.build()
    from paper_2509_16460_gb300 import ftcj
    return ftcj


CENTRES = np.array([[0.1, 0.2, 0.3], [1.9, 0.9, -0.4], [0.7, 3.1, 1.0], [-1.2, 1.0, 2.6]])


def device(w):
    import torch
    return torch.from_numpy(np.ascontiguousarray(w.Dk)).cuda()


@pytest.mark.parametrize("contraction", [0, 1])
def test_wide_contractions_in_split_plans(orc, F, contraction):
    """Two s and three d shells contracted over the same primitives: 17 functions per primitive, 289 outputs per
    record, above the 256 of the record-major maps.  The split form's bar, 1e-10 of max|J| (at least 1) as for the
    record-major maps."""
    import torch
    exps = np.array([0.15 * 1.5 ** q for q in range(12)])
    rng = np.random.default_rng(3)
    shells = [W.Shell(c, l, True, exps, rng.uniform(0.2, 0.8, 12)) for c in range(4) for l in (0, 0, 2, 2, 2)]
    nao = sum(s.nfunc for s in shells)
    Dk = W.random_bloch_density(rng, nao, (1, 1, 1), 3)[None]
    w = W.Workload("general-contraction", np.diag([11.0, 12.3, 11.6]), CENTRES, shells, (1, 1, 1), 0.42, Dk)
    ref = orc.lrj(w, want_j0n=False)
    plan = F.Plan.from_workload(w, precision=F.FTCJ_PREC_SPLIT, contraction=contraction)
    assert plan.info["contraction"] == F.FTCJ_CONTRACT_TC
    Jk, EJ = plan.jbuild(device(w))
    torch.cuda.synchronize()
    assert plan.status() == 0
    dJ = float(np.abs(Jk.cpu().numpy() - ref["Jk"]).max())
    scale = max(1.0, float(np.abs(ref["Jk"]).max()))
    dE = float(np.abs(EJ.cpu().numpy() - ref["EJ"]).max()) / max(1.0, float(np.abs(ref["EJ"]).max()))
    print(f"contraction {contraction}: records {plan.info['npairs']} max|dJ|={dJ:.2e} of {scale:.2e} rel dE={dE:.2e}")
    assert dJ <= 1e-10 * scale and dE <= 1e-10
    plan.close()


EVEN = [(c, l, [0.12 * 2.1 ** q for q in range(n)]) for c in range(4) for l, n in ((0, 9), (1, 5), (2, 2))]
DIFFUSE = [(c, l, [0.07, 0.4, 1.3]) for c in range(4) for l in (0, 1)]


def pair_of_densities(kind):
    """A cell whose passes run as sliced products in the named form, two densities, and the plan's arguments."""
    spec = DIFFUSE if kind == "classified" else EVEN
    w = W.tiny(seed=91, A=np.diag([11.0, 12.3, 11.6]), shell_spec=spec, kmesh=(1, 1, 1), omega=0.42, ndens=2,
               centres=CENTRES)
    args = {"fp64": dict(precision=0), "split": dict(precision=1), "tensor": dict(precision=1, contraction=1),
            "classified": dict(precision=0, classify=True)}[kind]
    return w, args


def touched(J):
    """The elements that some pair record contributes to."""
    return J != 0


KINDS = ["fp64", "split", "tensor", "classified"]


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("bad", [float("nan"), float("inf"), float("-inf")])
def test_a_non_finite_density_stays_non_finite(F, kind, bad):
    """One element of the first density is not finite: its E_J, J^k, rho and gradient show it, as the walks' do; the
    second density's results are those without it."""
    import torch
    w, args = pair_of_densities(kind)
    D = device(w)
    plan = F.Plan.from_workload(w, **args)
    assert plan.info["contraction"] == F.FTCJ_CONTRACT_TC
    J0, E0 = plan.jbuild(D)
    g0 = plan.grad(D)[1] if kind != "classified" else None
    D[0, 0, 3, 3] = bad
    J, E = plan.jbuild(D)
    torch.cuda.synchronize()
    assert plan.status() == 0
    assert not bool(torch.isfinite(E[0])) and not bool(torch.isfinite(J[0].real)[touched(J0[0])].any())
    scale = max(1.0, float(J0.abs().max()))
    assert float((J[1] - J0[1]).abs().max()) <= 1e-12 * scale and float((E[1] - E0[1]).abs()) <= 1e-12 * float(E0[1].abs())
    if g0 is not None:
        rho = plan.rho(plan.fold_density(D))
        assert not bool(torch.isfinite(rho[0].real).any()) and bool(torch.isfinite(rho[1].real).all())
        E2, g = plan.grad(D)
        assert not bool(torch.isfinite(E2[0])) and not bool(torch.isfinite(g[0]).any())
        assert float((g[1] - g0[1]).abs().max()) <= 1e-12 * max(1.0, float(g0.abs().max()))
        Wp = torch.ones((2, plan.ng_half), dtype=torch.complex128, device="cuda")
        Wp[0, 5] = bad
        J0n = plan.jback(Wp)
        assert not bool(torch.isfinite(J0n[0])[touched(J0n[1])].any()) and bool(torch.isfinite(J0n[1]).all())
    plan.close()


# FP64: any power of two that keeps E_J (quadratic) in FP64's range; split: double-float drops what lies below 2^-126,
# so one whose operands' last bits (2^-48, and W another 2^-14) lie above that
SCALES = {"fp64": (-300, -120, -90, 60, 300), "classified": (-300, -90, 300), "split": (-60, 40), "tensor": (-60, 40)}


@pytest.mark.parametrize("kind", KINDS)
def test_builds_scale_with_the_density(F, kind):
    """J(sD) = s J(D), E(sD) = s^2 E(D) and so on for powers of two s, in the first of two densities of a call, the
    second unscaled.  A power of two changes no significand, so the FP64 forms differ by the order of the atomic sums
    alone (1e-12 of max|J|); the split form's by what it drops below 2^-126 too (1e-10 of max|J|)."""
    import torch
    w, args = pair_of_densities(kind)
    D = device(w)
    plan = F.Plan.from_workload(w, **args)
    J0, E0 = plan.jbuild(D)
    g0 = plan.grad(D)[1] if kind != "classified" else None
    tol = 1e-12 if args["precision"] == 0 else 1e-10
    for e in SCALES[kind]:
        s = 2.0 ** e
        Ds = D.clone()
        Ds[0] *= s
        J, E = plan.jbuild(Ds)
        torch.cuda.synchronize()
        dJ = float((J[0] / s - J0[0]).abs().max()) / float(J0[0].abs().max())
        dE = float((E[0] / s / s - E0[0]).abs()) / float(E0[0].abs())
        d1 = float((J[1] - J0[1]).abs().max()) / float(J0[1].abs().max())
        print(f"{kind} 2^{e}: rel dJ={dJ:.2e} dE={dE:.2e} unscaled {d1:.2e}")
        assert dJ <= tol and dE <= tol and d1 <= 1e-12, (e, dJ, dE, d1)
        if g0 is not None:
            _, g = plan.grad(Ds)
            dg = float((g[0] / s / s - g0[0]).abs().max()) / float(g0[0].abs().max())
            assert dg <= tol * 10, (e, dg)
    plan.close()


@pytest.mark.parametrize("kind", KINDS)
def test_a_wait_that_gives_up_is_seen(F, kind, monkeypatch):
    """With a wait budget of 2 clock cycles the products give up and return: J^k and E_J are NaN, not what an earlier
    build left, the host call raises, and a batch reports it.  The next plan on the same GPU builds as before."""
    import torch
    w, args = pair_of_densities(kind)
    D = device(w)
    good = F.Plan.from_workload(w, **args)
    J0, E0 = good.jbuild(D)
    plan = F.Plan.from_workload(w, tc_wait_log2=1, **args)
    J, E = plan.jbuild(D)
    torch.cuda.synchronize()
    assert not bool(torch.isfinite(E).any()) and not bool(torch.isfinite(J.real)[touched(J0)].any())
    assert plan.status() & 1 and plan.status() == 0
    if kind != "classified":
        _, g = plan.grad(D)
        assert not bool(torch.isfinite(g).any()) and plan.status() & 1
    with pytest.raises(F.FtcjError, match="timed out"):
        plan.jbuild_host(w.Dk)
    assert plan.status() == 0
    plan.close()
    if kind == "fp64":
        params = F._params_of

        def impatient(*a, **k):
            p = params(*a, **k)
            p.tc_wait_log2 = 1
            return p

        monkeypatch.setattr(F, "_params_of", impatient)
        batch = F.Batch([w, w])
        assert batch.infos[0]["contraction"] == F.FTCJ_CONTRACT_TC
        batch.jbuild([D, D])
        with pytest.raises(F.FtcjError, match="timed out"):
            batch.status()
        assert batch.status() == 0
        batch.close()
    J, E = good.jbuild(D)
    torch.cuda.synchronize()
    assert good.status() == 0 and float((J - J0).abs().max()) <= 1e-12 * max(1.0, float(J0.abs().max()))
    good.close()
