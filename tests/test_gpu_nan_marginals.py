"""Memory strengths that overflow lambda to NaN: the faults are not decided and their messages
ignored, as in the oracle, wherever a fault sits (packed records, the general path, binary16
messages, the resuming launches, the plain kernel)."""
import numpy as np
import pytest

from oracle.relay import RelayParams, dmem_trace, relay_decode
from workloads import BB144, DecodingProblem, pack_bits, phenomenological_dem

from _cases import assert_same_decisions, gamma_for, gpu_decode, shots, syndrome

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
from paper_2511_21660_gb300 import (QLDPC_KERNEL_BASELINE, QLDPC_MSG_FP16,  # noqa: E402
                                    QLDPC_MSG_FP32, RelayConfig, RelayDecoder)

PREC = {QLDPC_MSG_FP32: "f32", QLDPC_MSG_FP16: "f16s"}


def _graph(M, N, degrees, dc):
    rng = np.random.default_rng(M * 1000 + N)
    H = np.zeros((M, N), dtype=np.uint8)
    for j in range(N):
        room = np.nonzero(H.sum(1) < dc)[0]
        H[rng.choice(room, min(int(rng.choice(degrees)), room.size), replace=False), j] = 1
    p = rng.uniform(0.005, 0.08, N)
    P = DecodingProblem("random", H, np.zeros((1, N), np.uint8), p, {"code": "bb72"})
    sig = syndrome(P, (rng.random((120, N)) < p).astype(np.uint8))
    sig[:20] = rng.random((20, M)) < 0.5
    return P, sig


def _strengths(P, R):
    """(1 - gamma) lambda(0) = -inf and gamma Lambda = +inf in the first iteration, in every
    leg for some of the faults."""
    gam = gamma_for(P, R=R, seed=P.N)
    rng = np.random.default_rng(P.N)
    gam[:, rng.random(P.N) < 0.04] = 3e38
    gam[1:, rng.random(P.N) < 0.04] = -3e38
    return gam


# whole warps of degree 2 and 3, ragged; mixed degrees; the families with 8 slots a fault
GRAPHS = [(160, 384, (2, 3), 8), (161, 391, (3,), 8), (130, 301, (0, 1, 2, 3, 4), 8),
          (120, 416, (2, 3), 16), (60, 351, (1, 2, 3, 5, 8), 32)]
CFG = dict(legs_after_first=6, iters_first=20, iters_later=15, stop_after_solutions=3)


@pytest.mark.parametrize("M,N,degrees,dc", GRAPHS)
@pytest.mark.parametrize("prec,clip", [(QLDPC_MSG_FP32, 0.0), (QLDPC_MSG_FP32, 12.0),
                                       (QLDPC_MSG_FP16, 0.0), (QLDPC_MSG_FP16, 12.0)])
def test_overflowing_strengths_match_the_mirror(M, N, degrees, dc, prec, clip):
    P, sig = _graph(M, N, degrees, dc)
    gam = _strengths(P, 6)
    prm = RelayParams(**CFG)
    if clip:
        prm.clip = clip
    ref = relay_decode(P.row_ptr, P.col_idx, P.p, gam, sig, prm, precision=PREC[prec],
                       want_marginals=True)
    assert np.isnan(ref.final_marginals).any() and (ref.legs > 1).any()
    for tail in (-1, 1):
        got = gpu_decode(P, gam, sig, RelayConfig(msg_precision=prec, llr_clip=clip,
                                                  tail_cut_iters=tail, **CFG))
        assert_same_decisions(got, ref, f"{M}x{N}/{PREC[prec]}/{clip}/{tail}")
    if prec == QLDPC_MSG_FP32:
        got = gpu_decode(P, gam, sig, RelayConfig(llr_clip=clip, kernel=QLDPC_KERNEL_BASELINE,
                                                  **CFG))
        assert_same_decisions(got, ref, "plain kernel")


@pytest.mark.parametrize("prec", [QLDPC_MSG_FP32, QLDPC_MSG_FP16])
def test_split_resuming_launch_keeps_nan(prec):
    P = phenomenological_dem(BB144, 11, 0.02)
    P.meta["code"] = "bb144"
    sig = shots(P, 60, 3)[1]
    gam = _strengths(P, 6)
    gam[0] = 0.125
    ref = relay_decode(P.row_ptr, P.col_idx, P.p, gam, sig, RelayParams(**CFG),
                       precision=PREC[prec])
    got = gpu_decode(P, gam, sig, RelayConfig(msg_precision=prec, tail_cut_iters=1, **CFG))
    assert (got[1] > 1).any()
    assert_same_decisions(got, ref, "split")


@pytest.mark.parametrize("prec", [QLDPC_MSG_FP32, QLDPC_MSG_FP16])
def test_recorded_marginals_are_nan_where_the_oracles_are(prec):
    P, sig = _graph(130, 301, (0, 1, 2, 3, 4), 8)
    gam = _strengths(P, 0)
    dec = RelayDecoder(P.row_ptr, P.col_idx, P.p, gam,
                       RelayConfig(legs_after_first=0, msg_precision=prec))
    out = dec.trace_first_leg(torch.from_numpy(pack_bits(sig[:16]).view(np.int64)).cuda(), 6)
    torch.cuda.synchronize()
    dec.close()
    ref = dmem_trace(P.row_ptr, P.col_idx, P.p, gam[0], sig[:16], 6, precision=PREC[prec])
    assert np.isnan(ref[0]).any() and np.isnan(ref[1]).any()
    for a, b in zip(out, ref):
        assert np.array_equal(a.cpu().numpy().transpose(1, 0, 2), b, equal_nan=True)
