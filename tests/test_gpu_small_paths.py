"""Paths chosen by the size of a cell or of its k-mesh: the FP64 mesh transforms
over lengths 1 to 6 (real ends, half-space of the unfold), the walks of cells of
few tiles (short chunks), and FP64 walks with and without their line table."""
import dataclasses

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


@pytest.mark.parametrize("kmesh", [(1, 1, 2), (3, 1, 1), (3, 3, 1), (1, 4, 1), (2, 3, 4), (4, 4, 4), (5, 1, 3),
                                   (3, 6, 1), (6, 2, 5), (5, 5, 1)])
def test_fp64_fold_and_unfold(orc, F, kmesh):
    """Both directions for inputs without any symmetry.  A value passes three
    axes of at most 6 terms, under 32 roundings of 2^-53 of its column's sum:
    2^-47 of that sum covers both sides."""
    import torch
    w = W.tiny(seed=35, A=np.diag([4.3, 4.6, 4.9]), kmesh=kmesh, ndens=2)
    plan = F.Plan.from_workload(w)
    rng = np.random.default_rng(17)
    shape = w.Dk.shape
    scale = 10.0 ** rng.uniform(-30, 3, size=shape[:1] + (1,) + shape[2:])
    Dk = (rng.normal(size=shape) + 1j * rng.normal(size=shape)) * scale
    got = plan.fold_density(torch.from_numpy(np.ascontiguousarray(Dk)).cuda()).cpu().numpy()
    ref = orc.fold_density(dataclasses.replace(w, Dk=Dk)).real
    assert (np.abs(got - ref) <= 2.0 ** -47 * np.abs(Dk).max(axis=1, keepdims=True)).all()
    J0n = rng.normal(size=got.shape) * scale
    Jk = plan.unfold_j(torch.from_numpy(np.ascontiguousarray(J0n)).cuda()).cpu().numpy()
    nd, nk, n, _ = J0n.shape
    Jref = (np.fft.ifftn(J0n.reshape(nd, *kmesh, n, n), axes=(1, 2, 3)) * nk).reshape(nd, nk, n, n)
    assert (np.abs(Jk - Jref) <= 2.0 ** -47 * nk * np.abs(J0n).max(axis=1, keepdims=True)).all()
    plan.close()


TRI = np.array([[0.0, 0.0, 0.0], [0.4, 0.0, 0.0], [-0.5, 0.3, 0.0]])


# a compact cell (short chunks, line table) and one whose lines hold more than
# the 32 points that a table may have (the recurrences)
@pytest.mark.parametrize("edges,omega", [((4.6, 5.2, 5.9), 0.37), ((60.0, 4.1, 4.4), 0.45)])
def test_triclinic_walks_against_the_oracle(orc, F, edges, omega):
    """J and E_J at the forms' own bounds (1e-10 and 1e-8 Eh), also with one
    chunk over the whole sphere."""
    import torch
    w = W.tiny(seed=71, A=np.diag(edges) + TRI, kmesh=(1, 2, 1), omega=omega, ndens=2)
    ref = orc.lrj(w, want_j0n=False)
    Dk = torch.from_numpy(np.ascontiguousarray(w.Dk)).cuda()
    for precision, tol in ((F.FTCJ_PREC_FP64, 1e-10), (F.FTCJ_PREC_SPLIT, 1e-8)):
        for chunk in (0, 4096):
            plan = F.Plan.from_workload(w, precision=precision, chunk_points=chunk)
            Jk, EJ = plan.jbuild(Dk)
            torch.cuda.synchronize()
            dJ = float(np.abs(Jk.cpu().numpy() - ref["Jk"]).max())
            dE = float(np.abs(EJ.cpu().numpy() - ref["EJ"]).max())
            print(f"edges {edges} precision {precision} chunk {chunk}: max|dJ|={dJ:.2e} max|dE|={dE:.2e}")
            assert dJ <= tol and dE <= tol * max(1.0, float(np.abs(ref["EJ"]).max()))
            plan.close()


@pytest.mark.parametrize("centres,exps", [(1, [0.4]), (2, [0.5, 1.4]), (7, [0.6])])
def test_gradient_assembly_over_few_and_many_centres(orc, F, centres, exps):
    """Blocks of 32 records: fewer than 32, more than four centres within a warp, a ragged last block.  Bar: FP64
    sums of up to 1e4 terms, 1e-10 of max|dE/dR| (at least 1)."""
    import torch
    rng = np.random.default_rng(centres)
    spec = [(c, l, exps) for c in range(centres) for l in ((0, 2) if c % 2 else (0, 1))]
    w = W.tiny(seed=70 + centres, A=np.array([[5.0, 0.0, 0.0], [0.6, 5.4, 0.0], [-0.3, 0.8, 5.2]]), shell_spec=spec,
               centres=(rng.random((centres, 3)) * 4.0).tolist(), kmesh=(1, 2, 1), omega=0.4, ndens=2)
    ref = orc.grad(w)
    for precision in (F.FTCJ_PREC_FP64, F.FTCJ_PREC_SPLIT):
        plan = F.Plan.from_workload(w, precision=precision)
        _, grad = plan.grad(torch.from_numpy(np.ascontiguousarray(w.Dk)).cuda())
        torch.cuda.synchronize()
        err = float(np.abs(grad.cpu().numpy() - ref).max())
        print(f"{centres} centres precision {precision}: records {plan.info['npairs']} max|dgrad|={err:.2e}")
        assert err <= 1e-10 * max(1.0, float(np.abs(ref).max()))
        plan.close()


def test_rows_of_partial_sums_of_a_long_sphere(F):
    """Few tiles over many chunks: a walk block per tile as long as the partial rows, each as long as the sphere, stay
    within 128 MB; the same J as from two blocks (the form's 1e-8 of max|J|)."""
    import torch
    spec = [(c, l, [0.2 * 1.15 ** q for q in range(n)]) for c in range(12) for l, n in ((0, 14), (1, 8), (2, 4))]
    w = W.tiny(seed=77, A=np.diag([30.0, 32.0, 34.0]) + 4.0 * TRI, shell_spec=spec, omega=0.5, eps_g=1e-30,
               centres=[[1.7 * i, 1.9 * j, 0.3 * (i + j)] for i in range(4) for j in range(3)])
    Dk = torch.from_numpy(np.ascontiguousarray(w.Dk)).cuda()
    got = []
    for blocks in (0, 2):
        plan = F.Plan.from_workload(w, precision=F.FTCJ_PREC_SPLIT, rho_blocks=blocks)
        info = plan.info
        if not blocks:
            tiles = sum(-(-n // 128) for n in info["pairs_by_class"])
            print(f"points {info['ng_half']} chunks {info['nchunks']} tiles {tiles} blocks {info['rho_blocks']}")
            assert info["nchunks"] > 100 and info["rho_blocks"] * info["ng_half"] * 16 <= 128 << 20
            assert info["rho_blocks"] < tiles
        got.append(plan.jbuild(Dk)[0])
        torch.cuda.synchronize()
        plan.close()
    assert float((got[0] - got[1]).abs().max()) <= 1e-8 * max(1.0, float(got[1].abs().max()))
