"""Plans made while device memory is short: the product's operand workspace is
used in several passes, and a plan that does not fit with products runs the walks."""
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


def leave_free(nbytes):
    """Holds device memory so that about nbytes stay free."""
    import torch
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    assert free > nbytes
    return torch.empty(free - nbytes, dtype=torch.uint8, device="cuda")


def test_plans_under_short_memory(F):
    """The molecular crystal in the FP64 form.  With 8 GB free its operand tiles take several passes; with little more
    than the walks need it falls back to them.  J^k is the same in all cases (the forms' 1e-12 of max|J|)."""
    import torch
    w = W.cfg3()
    D = torch.from_numpy(np.ascontiguousarray(w.Dk)).cuda()
    out = [(torch.empty_like(D), torch.empty(w.ndens, dtype=torch.float64, device="cuda")) for _ in range(2)]
    product, walk = F.Plan.from_workload(w), F.Plan.from_workload(w, chunk_points=4096)
    assert (product.info["contraction"], product.info["rho_walk_launches"]) == (F.FTCJ_CONTRACT_TC, 2)
    need = walk.info["device_bytes"]
    print(f"device bytes: product {product.info['device_bytes']} walk {need}")
    ref, _ = product.jbuild(D, *out[0])
    walk.jbuild(D, *out[1])
    torch.cuda.synchronize()
    product.close()
    walk.close()
    tol = 1e-12 * max(1.0, float(ref.abs().max()))
    assert float((out[1][0] - ref).abs().max()) <= tol
    seen = set()
    for extra in [8 << 30] + [(96 << 20) * k for k in (1, 2, 4, 8)]:
        hold = leave_free(extra if extra == 8 << 30 else need + extra)
        plan = F.Plan.from_workload(w)
        J, _ = plan.jbuild(D, *out[1])
        torch.cuda.synchronize()
        info = plan.info
        plan.close()
        del hold
        torch.cuda.empty_cache()
        print(f"extra {extra >> 20} MB: contraction {info['contraction']} launches {info['rho_walk_launches']} "
              f"bytes {info['device_bytes']}")
        seen.add((info["contraction"], info["rho_walk_launches"] > 2))
        assert float((J - ref).abs().max()) <= tol
    assert {(F.FTCJ_CONTRACT_TC, True), (F.FTCJ_CONTRACT_WALK, False)} <= seen, seen
