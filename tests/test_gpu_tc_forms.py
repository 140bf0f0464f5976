"""The separable contraction's layouts against the FP64 oracle, in the FP64
form (eight slices) and the split tensor-core form: odd and even numbers of
axis points per slot group, one and several row tiles, one and several slot
parts, wide and narrow column counts, density groups that do not divide.

Bars.  FP64 form: every operand is within 2^-55 of its row's or column's bound
and every level sum is exact, so an output of K terms is within K 2^-54 of the
bounds; with K below 2^12 records and slots here that is 2^-42, and 1e-12 of
max|J| (at least 1) leaves room for the FP64 steps around it.  Split form: the
form's own 1e-8 Eh."""
import numpy as np
import pytest

from paper_2509_16460_gb300 import workloads as W

pytestmark = pytest.mark.gpu

SPD = [(0, 0, [0.3, 1.7]), (0, 1, [0.6]), (1, 0, [0.45]), (1, 2, [0.8])]
SP = [(0, 0, [0.25, 2.0]), (1, 0, [0.5]), (1, 1, [0.7])]

#       edges              shells kmesh      omega  ndens
CELLS = [
    ([4.1, 4.4, 4.9], SPD, (1, 1, 1), 0.30, 1),    # a handful of points: one window per class, one tile
    ([5.0, 6.1, 7.3], SPD, (2, 1, 1), 0.45, 3),    # three densities
    ([4.3, 4.3, 15.0], SP, (1, 1, 2), 0.40, 2),    # a long axis: many columns or many rows
    ([13.0, 12.1, 12.6], SP, (1, 2, 1), 0.50, 1),  # several row tiles, two slot parts in the FP64 form
    ([22.0, 18.0, 5.0], SP, (1, 1, 1), 0.50, 2),   # more than 1024 slots or wide columns
]


@pytest.fixture(scope="module")
def F():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2509_16460_gb300 import build
    build.build()
    from paper_2509_16460_gb300 import ftcj
    return ftcj


def cell(index):
    edges, spec, kmesh, omega, ndens = CELLS[index]
    return W.tiny(seed=60 + index, A=np.diag(edges), centres=[[0.1, 0.2, 0.3], [1.3, 0.9, -0.4]], shell_spec=spec,
                  kmesh=kmesh, omega=omega, ndens=ndens)


@pytest.mark.parametrize("index", range(len(CELLS)))
def test_contraction_layouts(orc, F, index):
    import torch
    w = cell(index)
    ref = orc.lrj(w, want_j0n=False)
    scale = max(1.0, float(np.abs(ref["Jk"]).max()))
    Dk = torch.from_numpy(np.ascontiguousarray(w.Dk)).cuda()
    for precision, contraction, tol in ((F.FTCJ_PREC_FP64, F.FTCJ_CONTRACT_WALK, 1e-12 * scale),
                                        (F.FTCJ_PREC_SPLIT, F.FTCJ_CONTRACT_TC, 1e-8)):
        plan = F.Plan.from_workload(w, precision=precision, contraction=contraction)
        try:
            assert plan.info["contraction"] == F.FTCJ_CONTRACT_TC
            Jk, EJ = plan.jbuild(Dk)
            # fewer densities than the plan holds
            J1, E1 = plan.jbuild(Dk[-1:].contiguous())
            torch.cuda.synchronize()
            assert plan.status() == 0
            dJ = float(np.abs(Jk.cpu().numpy() - ref["Jk"]).max())
            dE = float((np.abs(EJ.cpu().numpy() - ref["EJ"]) / np.maximum(1.0, np.abs(ref["EJ"]))).max())
            d1 = float(np.abs(J1.cpu().numpy() - ref["Jk"][-1:]).max())
            print(f"cell {index} precision {precision}: max|dJ|={dJ:.2e} rel dE={dE:.2e} single {d1:.2e} "
                  f"rows {plan.info['tc_rows']} tiles {plan.info['tc_row_tiles']} blocks {plan.info['tc_blocks_per_window']}")
            assert dJ <= tol and d1 <= tol and dE <= tol, (index, precision, dJ, d1, dE)
        finally:
            plan.close()


def test_fp64_walks_agree_with_contraction(F):
    """A caller's own walk shape keeps the FP64 walks; both give the same J^k."""
    import torch
    w = cell(1)
    Dk = torch.from_numpy(np.ascontiguousarray(w.Dk)).cuda()
    a = F.Plan.from_workload(w)
    b = F.Plan.from_workload(w, chunk_points=4096)
    assert (a.info["contraction"], b.info["contraction"]) == (F.FTCJ_CONTRACT_TC, F.FTCJ_CONTRACT_WALK)
    Ja, Ea = a.jbuild(Dk)
    Jb, Eb = b.jbuild(Dk)
    torch.cuda.synchronize()
    scale = max(1.0, float(Jb.abs().max()))
    assert float((Ja - Jb).abs().max()) <= 1e-12 * scale
    assert float(((Ea - Eb).abs() / Eb.abs().clamp_min(1.0)).max()) <= 1e-12
    a.close()
    b.close()


#       edges               kmesh      omega  ndens  taken
SPLIT_CELLS = [
    ([11.0, 12.3, 11.6], (1, 1, 1), 0.42, 1, True),
    ([9.1, 9.7, 18.0], (2, 1, 1), 0.45, 3, True),   # three densities, a long axis
    ([26.0, 10.0, 8.0], (1, 1, 1), 0.40, 2, True),  # odd counts of records and points
    ([6.3, 6.0, 5.7], (1, 2, 1), 0.40, 2, False),   # below 512 points: the walk
]
EVEN = [(c, l, [0.12 * 2.1 ** q for q in range(n)]) for c in range(4) for l, n in ((0, 9), (1, 5), (2, 2))]


@pytest.mark.parametrize("index", range(len(SPLIT_CELLS)))
def test_split_walk_plans_take_structure_factors_from_the_product(orc, F, index):
    """Above the size rule a split plan's rho comes from the eight-slice product and its J' from the walk; both
    against the oracle and a caller's own walk shape.  Bar: double-float steps of 2^-45, at most 40 along a chain
    (the walk), 1e-10 of max|J| (at least 1); the gradient likewise."""
    import torch
    edges, kmesh, omega, ndens, taken = SPLIT_CELLS[index]
    w = W.tiny(seed=90 + index, A=np.diag(edges), shell_spec=EVEN, kmesh=kmesh, omega=omega, ndens=ndens,
               centres=[[0.1, 0.2, 0.3], [1.9, 0.9, -0.4], [0.7, 3.1, 1.0], [-1.2, 1.0, 2.6]])
    ref = orc.lrj(w, want_j0n=False)
    scale = max(1.0, float(np.abs(ref["Jk"]).max()))
    Dk = torch.from_numpy(np.ascontiguousarray(w.Dk)).cuda()
    got = []
    for chunk in (0, 4096):
        plan = F.Plan.from_workload(w, precision=F.FTCJ_PREC_SPLIT, chunk_points=chunk)
        info = plan.info
        want = F.FTCJ_CONTRACT_TC if taken and not chunk else F.FTCJ_CONTRACT_WALK
        assert (info["contraction"], info["j_contraction"]) == (want, F.FTCJ_CONTRACT_WALK), info
        Jk, EJ = plan.jbuild(Dk)
        E2, grad = plan.grad(Dk)
        J1, _ = plan.jbuild(Dk[-1:].contiguous())  # fewer densities than the plan holds
        torch.cuda.synchronize()
        assert plan.status() == 0
        dJ = float(np.abs(Jk.cpu().numpy() - ref["Jk"]).max())
        d1 = float(np.abs(J1.cpu().numpy() - ref["Jk"][-1:]).max())
        dE = float((np.abs(EJ.cpu().numpy() - ref["EJ"]) / np.maximum(1.0, np.abs(ref["EJ"]))).max())
        print(f"cell {index} chunk {chunk}: records {info['npairs']} points {info['ng_half']} max|dJ|={dJ:.2e} "
              f"rel dE={dE:.2e}")
        assert dJ <= 1e-10 * scale and d1 <= 1e-10 * scale and dE <= 1e-10
        assert bool(torch.equal(E2, EJ))
        got.append((rho_of(plan, Dk), grad))
        plan.close()
    (ra, ga), (rb, gb) = got
    assert float((ra - rb).abs().max()) <= 1e-10 * max(1.0, float(rb.abs().max()))
    assert float((ga - gb).abs().max()) <= 1e-10 * max(1.0, float(gb.abs().max()))


def rho_of(plan, Dk):
    return plan.rho(plan.fold_density(Dk))


@pytest.mark.parametrize("index", range(len(CELLS)))
def test_gradient_sums_of_the_product(orc, F, index):
    """The degree-(L+1) sums of the FP64 form's gradient from the product, against the oracle and the walks.  Bar: the
    derivative's terms are at most 2 alpha n^5 times the build's, held to 2^-42 of their bounds as above; 1e-10 of
    max|dE/dR| (at least 1) leaves room for the cancellation between the two centres."""
    import torch
    w = cell(index)
    Dk = torch.from_numpy(np.ascontiguousarray(w.Dk)).cuda()
    ref = orc.grad(w)
    scale = max(1.0, float(np.abs(ref).max()))
    got = []
    for chunk in (0, 4096):
        plan = F.Plan.from_workload(w, chunk_points=chunk)
        _, grad = plan.grad(Dk)
        _, last = plan.grad(Dk[-1:].contiguous())  # fewer densities than the plan holds
        torch.cuda.synchronize()
        assert plan.status() == 0
        got.append(grad.cpu().numpy())
        err = float(np.abs(got[-1] - ref).max())
        print(f"cell {index} chunk {chunk}: max|dgrad|={err:.2e} of {scale:.2e}")
        assert err <= 1e-10 * scale
        assert float(np.abs(last.cpu().numpy() - ref[-1:]).max()) <= 1e-10 * scale
        plan.close()
    assert float(np.abs(got[0] - got[1]).max()) <= 1e-10 * scale


#       edges               omega  the sums' form
GRADIENT_CELLS = [([5.0, 6.1, 7.3], 0.45, "product"),
                  ([4.1, 4.4, 34.0], 0.50, "walk")]  # |n| up to 30: n^5 is not exact in FP32


@pytest.mark.parametrize("edges,omega,form", GRADIENT_CELLS)
def test_form_of_the_gradient_sums(orc, F, edges, omega, form):
    """Which form runs the degree-(L+1) sums, and that the structure factors' product with the walk's sums gives the
    oracle's gradient too (the bar of the product's, above)."""
    import torch
    w = W.tiny(seed=66, A=np.diag(edges), centres=[[0.1, 0.2, 0.3], [1.3, 0.9, -0.4]], shell_spec=SP, omega=omega)
    ref = orc.grad(w)
    plan, walk = F.Plan.from_workload(w), F.Plan.from_workload(w, chunk_points=4096)
    assert plan.info["contraction"] == F.FTCJ_CONTRACT_TC and walk.info["contraction"] == F.FTCJ_CONTRACT_WALK
    assert plan.info["grad_contraction"] == (F.FTCJ_CONTRACT_TC if form == "product" else F.FTCJ_CONTRACT_WALK)
    assert walk.info["grad_contraction"] == F.FTCJ_CONTRACT_WALK
    _, grad = plan.grad(torch.from_numpy(np.ascontiguousarray(w.Dk)).cuda())
    torch.cuda.synchronize()
    assert plan.status() == 0
    assert float(np.abs(grad.cpu().numpy() - ref).max()) <= 1e-10 * max(1.0, float(np.abs(ref).max()))
    plan.close()
    walk.close()
