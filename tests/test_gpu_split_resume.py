"""The resuming launch that spreads a shot over a cluster of blocks: the same results as the
single launch, with every shot moved at its first leg boundary, for graphs cut between rounds,
graphs whose faults reach across every cut, odd sizes, both precisions; and the oracle's on
sampled shots.  Batches small enough run all their records there (more records than clusters
take turns); a large one with more records than clusters runs the one-block launch."""
import numpy as np
import pytest

from oracle.relay import RelayParams, relay_decode
from workloads import BB72, BB144, BB288, DecodingProblem, phenomenological_dem

from _cases import assert_same_decisions, gamma_for, gpu_decode, shots, syndrome

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
from paper_2511_21660_gb300 import QLDPC_MSG_FP16, QLDPC_MSG_FP32, RelayConfig  # noqa: E402

PREC = {QLDPC_MSG_FP32: "f32", QLDPC_MSG_FP16: "f16s"}


def _check(P, sig, prec, few=25, **cfg):
    gam = gamma_for(P, R=cfg["legs_after_first"], seed=P.N)
    on = gpu_decode(P, gam, sig, RelayConfig(msg_precision=prec, tail_cut_iters=1, **cfg))
    off = gpu_decode(P, gam, sig, RelayConfig(msg_precision=prec, tail_cut_iters=-1, **cfg))
    for a, b in zip(on[:4], off[:4]):
        assert np.array_equal(a, b)
    hard = np.argsort(on[3])[-few:]
    assert (on[1][hard] > 1).all()                       # they went through the second launch
    ref = relay_decode(P.row_ptr, P.col_idx, P.p, gam, sig[hard], RelayParams(**cfg),
                       precision=PREC[prec])
    assert_same_decisions(tuple(x[hard] for x in on[:4]), ref, "resumed")


@pytest.mark.parametrize("code,rounds,n", [(BB72, 7, 300), (BB72, 7, 2500), (BB144, 11, 200),
                                           (BB144, 12, 90), (BB288, 18, 60)])
@pytest.mark.parametrize("prec", [QLDPC_MSG_FP32, QLDPC_MSG_FP16])
def test_detector_models(code, rounds, n, prec):
    P = phenomenological_dem(code, rounds, 0.02)
    P.meta["code"] = "bb288" if code is BB288 else "bb144"
    sig = shots(P, n, 3 + rounds)[1]
    _check(P, sig, prec, legs_after_first=12, iters_first=30, iters_later=20,
           stop_after_solutions=4)


@pytest.mark.parametrize("prec", [QLDPC_MSG_FP32, QLDPC_MSG_FP16])
@pytest.mark.parametrize("mode", [dict(), dict(warm_start_mode=1), dict(max_total_iters=77)])
def test_faults_across_every_cut_and_odd_sizes(prec, mode):
    rng = np.random.default_rng(12)
    M, N = 301, 701
    H = np.zeros((M, N), dtype=np.uint8)
    for j in range(N - 1):                               # the last fault has no check
        room = np.nonzero(H.sum(1) < 8)[0]
        H[rng.choice(room, min(int(rng.integers(1, 4)), room.size), replace=False), j] = 1
    p = rng.uniform(0.01, 0.06, N)
    P = DecodingProblem("across", H, np.zeros((1, N), np.uint8), p, {"code": "bb72"})
    sig = syndrome(P, (rng.random((150, N)) < p).astype(np.uint8))
    sig[:40] = rng.random((40, M)) < 0.5
    _check(P, sig, prec, legs_after_first=6, iters_first=20, iters_later=15,
           stop_after_solutions=3, **mode)
