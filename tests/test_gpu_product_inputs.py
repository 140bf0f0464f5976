"""What the sliced product has to take as the walks do: general contractions
with many functions per primitive."""
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
