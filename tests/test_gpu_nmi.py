"""GPU parity of the NMI map (CMIF_FLAG_NMI) against the oracle's
(H_A + H_B) / H_AB from the direct method's entropies.

Tolerance: each entropy of the fixed-point reduction is within ~1.1e-6 bits
(the MI bound), so |dNMI| <= (|dH_A| + |dH_B| + NMI |dH_AB|) / H_AB
<= 4.4e-6 / H_AB; the test allows 5e-6 / H_AB, and exact 0 where H_AB = 0.
"""
import numpy as np
import pytest

import oracle
import synth
from tolerances import MI_TOL

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cm():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2106_14699_gb300 as cm
    from paper_2106_14699_gb300 import build
    build.build()
    cm.lib()
    return cm


def _dev(x):
    return None if x is None else torch.from_numpy(np.ascontiguousarray(x)).to("cuda:0")


def _check(got, ref):
    hab = ref["h_ab"]
    zero = hab == 0
    assert np.all(got[zero] == 0.0)
    tol = 5e-6 / np.maximum(hab[~zero], 1e-300)
    err = np.abs(got[~zero] - ref["nmi"][~zero])
    assert np.all(err <= tol), float((err / tol).max())


@pytest.mark.parametrize("shape,K,prec", [
    ((150, 200), 8, "FP32"),     # TMEM row kernel (Q = 512)
    ((96, 520), 8, "FP32"),      # TMEM row kernel (Q = 2048)
    ((40, 1100), 6, "FP32"),     # TMEM row kernel, teams of three warps (Q = 3072)
    ((70, 66), 6, "FP64"),
    ((70, 66), 6, "SPLIT32"),
])
def test_nmi_map_vs_oracle(cm, shape, K, prec):
    rng = np.random.default_rng(sum(shape) + K)
    A = rng.integers(0, K, shape).astype(np.int32)
    A[: shape[0] // 2, : shape[1] // 3] = 2
    B = np.roll(A, (5, -9), axis=(0, 1))
    B[rng.random(B.shape) < 0.25] = 1
    MB = (rng.random(B.shape) > 0.1).astype(np.uint8)
    H, W = shape
    R, C = 2 * H - 1, 2 * W - 1
    plan = cm.Plan(H, W, H, W, K, K, getattr(cm, prec), nmi=True)
    m = torch.empty((R, C), dtype=torch.float64, device="cuda:0")
    n = torch.empty((R, C), dtype=torch.int32, device="cuda:0")
    pk = torch.empty(24, dtype=torch.uint8, device="cuda:0")
    plan.compute(_dev(A), None, _dev(B), _dev(MB), m, n, None, 0.5, pk)
    assert plan.status()[0] == "OK"
    ref = oracle.nmi(A, None, B, MB, K, K)
    got = m.cpu().numpy()
    _check(got, ref)
    assert np.array_equal(n.cpu().numpy(), ref["n"])
    # Alg. 1 on the NMI map: the peak is the gated argmax of NMI
    idx, v, nn = oracle.gamma_argmax(ref["nmi"], ref["n"], 0.5)
    a, dy, dx, gn, gv = cm.peaks_from_bytes(pk, 1)[0]
    assert abs(gv - v) <= 5e-6 / max(ref["h_ab"].flat[idx], 1e-3)
    plan.close()


def test_nmi_single256_full_map(cm):
    cfg = synth.make_workload("single-256x256-K16")
    A, B, MA, MB = cfg["A"], cfg["B"], cfg["M_A"], cfg["M_B"]
    H, W = A.shape
    plan = cm.Plan(H, W, H, W, 16, 16, cm.FP32, nmi=True)
    m = torch.empty((2 * H - 1, 2 * W - 1), dtype=torch.float64, device="cuda:0")
    plan.compute(_dev(A), _dev(MA), _dev(B), _dev(MB), m)
    assert plan.status()[0] == "OK"
    _check(m.cpu().numpy(), oracle.nmi(A, MA, B, MB, 16, 16))
    plan.close()


@pytest.mark.parametrize("W,KB", [(1100, 8), (1100, 7), (1100, 6), (1100, 5), (700, 17), (700, 16)])
def test_few_rows_near_the_shared_memory_limit(cm, W, KB):
    """Maps of few, wide rows with count maps (generic row kernel, Q = 3072 and 1536): a cluster
    of blocks per row where its partial sums fit beside the B-marginals (MI: up to 7 labels at
    3072; NMI: up to 5, and up to 16 at 1536), else one block per row.  MI, NMI, N and every
    count against the oracle."""
    rng = np.random.default_rng(W + KB)
    A = rng.integers(0, 4, (30, W)).astype(np.int32)
    B = rng.integers(0, KB, (30, W - 3)).astype(np.int32)
    MB = (rng.random(B.shape) > 0.1).astype(np.uint8)
    ref = oracle.cmif(A, None, B, MB, 4, KB, counts=True, marginals=True)
    R, C = ref["mi"].shape
    for nmi in (False, True):
        plan = cm.Plan(*A.shape, *B.shape, 4, KB, cm.FP32, nmi=nmi, debug_counts=True)
        m = torch.empty((R, C), dtype=torch.float64, device="cuda:0")
        n = torch.empty((R, C), dtype=torch.int32, device="cuda:0")
        counts = torch.empty((4 * KB + 4 + KB, R, C), dtype=torch.int32, device="cuda:0")
        plan.compute(_dev(A), None, _dev(B), _dev(MB), m, n, counts)
        assert plan.status()[0] == "OK"
        plan.close()
        assert np.array_equal(n.cpu().numpy(), ref["n"])
        got = counts.cpu().numpy()
        assert np.array_equal(got, np.concatenate([ref["joint"], ref["marg_a"], ref["marg_b"]]))
        if nmi:
            _check(m.cpu().numpy(), oracle.nmi(A, None, B, MB, 4, KB))
        else:
            assert float(np.abs(m.cpu().numpy() - ref["mi"]).max()) <= MI_TOL


@pytest.mark.parametrize("prec", ["FP64", "SPLIT32"])
def test_few_rows_exact_nmi(cm, prec):
    """The same limit of the exact plans: NMI at Q = 2048 with one label b, whose row takes
    200 KB without a cluster's partial sums."""
    rng = np.random.default_rng(9)
    A = rng.integers(0, 3, (20, 620)).astype(np.int32)
    B = np.zeros((25, 600), np.int32)
    MB = (rng.random(B.shape) > 0.3).astype(np.uint8)
    plan = cm.Plan(*A.shape, *B.shape, 3, 1, getattr(cm, prec), nmi=True)
    m = torch.empty((plan.R, plan.C), dtype=torch.float64, device="cuda:0")
    plan.compute(_dev(A), None, _dev(B), _dev(MB), m)
    assert plan.status()[0] == "OK"
    plan.close()
    _check(m.cpu().numpy(), oracle.nmi(A, None, B, MB, 3, 1))
