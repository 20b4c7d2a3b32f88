"""The all-of-K GEMM's two kernels, for rows of A, B and C that are all 16-byte
aligned with whole sixteens of K, and for any rows: each condition broken in
turn.  Tolerance: the FP32 summation bound of the product, (K + 4) 2^-23 of the
sum of absolute terms, as for the other GEMM shapes."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# K, then offset of the first element and padding of a row of A, B, C; beta; atomic
CASES = [(64, 0, 0, 0, 0, 0, 0, 0.0, False), (64, 0, 0, 0, 0, 0, 0, 0.5, False), (64, 0, 8, 0, 16, 0, 4, 0.0, False),
         (64, 1, 0, 0, 0, 0, 0, 0.0, False), (64, 0, 0, 8, 0, 0, 0, 0.0, False), (64, 0, 0, 3, 0, 0, 0, 0.0, False),
         (64, 0, 1, 0, 0, 0, 0, 0.0, False), (64, 0, 0, 0, 4, 0, 0, 0.0, False), (64, 0, 0, 0, 0, 1, 0, 0.5, False),
         (64, 0, 0, 0, 0, 0, 1, 0.5, False), (40, 0, 0, 0, 0, 0, 0, 0.0, False), (17, 0, 0, 0, 0, 0, 0, 0.0, False),
         (256, 0, 0, 0, 0, 0, 0, 0.0, False), (255, 0, 1, 0, 1, 0, 0, 0.0, False), (16, 0, 0, 0, 0, 0, 0, 0.0, True)]


@pytest.mark.parametrize("N", [16, 44, 64, 160])
@pytest.mark.parametrize("case", CASES, ids=["-".join(map(str, c)) for c in CASES])
def test_gemm_rows_of_any_alignment(case, N):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1406_7459_gb300 import mm
    K, oa, pa, ob, pb, oc, pc, beta, atomic = case
    M = 200
    rng = np.random.default_rng(K * 1000 + N)

    def buffer(rows, row, off, dtype):
        x = torch.from_numpy(rng.standard_normal(off + rows * row).astype(np.float32)).to(dtype)
        return x.cuda(), x[off:].double().numpy().reshape(rows, row)

    A, a = buffer(M, K + pa, oa, torch.bfloat16)
    B, b = buffer(N, K + pb, ob, torch.bfloat16)
    C, c = buffer(M, N + pc, oc, torch.float32)
    a, b = a[:, :K], b[:, :K]
    mm.mm_gemm_bf16(A[oa:], B[ob:], C[oc:], M, N, K, (K + pa, 1, 1, K + pb, N + pc, 1), alpha=0.5, beta=beta,
                    atomic=atomic)
    old = c[:, :N] * (1.0 if atomic else beta)
    want = 0.5 * a @ b.T + old
    bound = (K + 4) * 2.0 ** -23 * (0.5 * np.abs(a) @ np.abs(b).T + np.abs(old)) + 1e-30
    got = C.cpu()[oc:].double().numpy().reshape(M, N + pc)
    assert np.all(np.abs(got[:, :N] - want) <= bound)
    assert np.array_equal(got[:, N:], c[:, N:])              # nothing written past a row
