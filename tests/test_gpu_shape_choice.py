"""The shape the library takes for graphs with more checks than its codes have for their faults,
and the results there."""
import numpy as np
import pytest

from oracle.relay import RelayParams, relay_decode
from workloads import DecodingProblem

from _cases import assert_same_decisions, gamma_for, gpu_decode, syndrome

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
from paper_2511_21660_gb300 import QLDPC_MSG_FP16, QLDPC_MSG_FP32, RelayConfig  # noqa: E402

PREC = {QLDPC_MSG_FP32: "f32", QLDPC_MSG_FP16: "f16s"}


def _problem(M, N, dc, seed):
    """Degree 2 and 3, rows dealt evenly but for one full row."""
    rng = np.random.default_rng(seed)
    H = np.zeros((M, N), dtype=np.uint8)
    H[0, :dc] = 1
    rows = 1 + np.concatenate([rng.permutation(M - 1) for _ in range(3 * N // (M - 1) + 1)])
    k = 0
    for j in range(dc, N):
        d = int(rng.integers(2, 4))
        H[rows[k:k + d], j] = 1
        k += d
    assert H.sum(1).max() == dc and 1 <= H.sum(0).max() <= 4
    return DecodingProblem("rows", H, np.zeros((1, N), np.uint8), np.full(N, 0.01),
                           {"code": "bb72"})


# (checks, faults, row slots, precision, threads): messages above 64 KB take the first shape with
# records in messages; shared memory for few narrow blocks takes the wide shape; just below the
# line the narrow shape stays
CASES = [(2100, 1500, 8, QLDPC_MSG_FP32, 640), (1040, 900, 16, QLDPC_MSG_FP32, 640),
         (2100, 1000, 16, QLDPC_MSG_FP16, 640), (800, 700, 8, QLDPC_MSG_FP32, 256),
         (1900, 1500, 8, QLDPC_MSG_FP32, 512), (3600, 3500, 8, QLDPC_MSG_FP32, 1024),
         (2600, 3500, 8, QLDPC_MSG_FP32, 256), (300, 700, 8, QLDPC_MSG_FP32, 64)]


@pytest.mark.parametrize("M,N,dc,prec,threads", CASES)
def test_shape_and_results(M, N, dc, prec, threads):
    P = _problem(M, N, dc, M + N)
    rng = np.random.default_rng(4)
    few = 40
    sig = syndrome(P, (rng.random((few, N)) < P.p).astype(np.uint8))
    sig[:5] = rng.random((5, M)) < 0.5
    sig = np.concatenate([sig, sig[rng.integers(0, few, 8000 - few)]])   # above any small batch
    gam = gamma_for(P, R=3, seed=1)
    cfg = dict(legs_after_first=3, iters_first=15, iters_later=10, stop_after_solutions=2)
    got = gpu_decode(P, gam, sig, RelayConfig(msg_precision=prec, **cfg))
    assert got[4].block_threads == threads
    ref = relay_decode(P.row_ptr, P.col_idx, P.p, gam, sig[:few], RelayParams(**cfg),
                       precision=PREC[prec])
    assert_same_decisions(tuple(x[:few] for x in got[:4]), ref, f"{M}x{N}/{dc}")
    wide = gpu_decode(P, gam, sig, RelayConfig(msg_precision=prec, block_threads=1024, **cfg))
    for a, b in zip(got[:4], wide[:4]):
        assert np.array_equal(a, b)
