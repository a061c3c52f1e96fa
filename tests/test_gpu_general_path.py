"""Faults of degree 2 and 3 that have no packed slot record: graphs with more than 64 KB of
messages and at most 3072 faults, in the families with 4 and with 8 slots a fault, alone and in
warps with other degrees; against the oracle mirror bit for bit, in every block size."""
import numpy as np
import pytest

from oracle.relay import RelayParams, relay_decode
from workloads import DecodingProblem

from _cases import assert_same_decisions, gamma_for, gpu_decode, syndrome

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
from paper_2511_21660_gb300 import (QLDPC_MSG_FP16, QLDPC_MSG_FP32, QldpcError,  # noqa: E402
                                    RelayConfig)


def _graph(M, N, degrees, dc, seed):
    rng = np.random.default_rng(seed)
    H = np.zeros((M, N), dtype=np.uint8)
    H[0, :dc] = 1                                   # a full row: fixes the family
    for j in range(dc, N):
        d = int(rng.choice(degrees))
        H[rng.choice(np.arange(1, M), d, replace=False), j] = 1
    assert H.sum(1).max() == dc
    return H


# (checks, faults, degrees, check degree, precision): just above 64 KB of messages
CASES = [(1040, 700, (2, 3), 16, QLDPC_MSG_FP32), (1040, 701, (2, 3, 6), 16, QLDPC_MSG_FP32),
         (520, 500, (2, 3), 32, QLDPC_MSG_FP32), (2080, 900, (2, 3), 16, QLDPC_MSG_FP16),
         (2080, 1500, (2, 3), 8, QLDPC_MSG_FP32)]


@pytest.mark.parametrize("M,N,degrees,dc,prec", CASES)
def test_degree_two_and_three_without_records(M, N, degrees, dc, prec):
    H = _graph(M, N, degrees, dc, M + N)
    p = np.full(N, 0.01)
    P = DecodingProblem("tall", H, np.zeros((1, N), np.uint8), p, {"code": "bb72"})
    rng = np.random.default_rng(3)
    sig = syndrome(P, (rng.random((60, N)) < p).astype(np.uint8))
    sig[:8] = rng.random((8, M)) < 0.5
    gam = gamma_for(P, R=4, seed=1)
    cfg = dict(legs_after_first=4, iters_first=15, iters_later=10, stop_after_solutions=2)
    ref = relay_decode(P.row_ptr, P.col_idx, P.p, gam, sig, RelayParams(**cfg),
                       precision={QLDPC_MSG_FP32: "f32", QLDPC_MSG_FP16: "f16s"}[prec])
    ran = 0
    for bt in (0, 256, 512, 1024):
        try:
            got = gpu_decode(P, gam, sig, RelayConfig(msg_precision=prec, block_threads=bt, **cfg))
        except QldpcError:                          # no shape of that size holds the graph
            continue
        assert_same_decisions(got, ref, f"{M}x{N}/{dc}/{bt}")
        ran += 1
    assert ran >= 3
