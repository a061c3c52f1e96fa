"""Paths of the decode kernels' check and fault passes, against the oracle mirror bit for bit:
packed slot records and the general fault path in one warp, rows with no, one or several
padding slots, saturated messages, and the recorded messages of the first leg."""
import numpy as np
import pytest

from oracle.relay import RelayParams, dmem_trace, relay_decode
from workloads import BB72, BB144, BB288, DecodingProblem, pack_bits, phenomenological_dem

from _cases import assert_same_decisions, gamma_for, gpu_decode, shots, syndrome

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
from paper_2511_21660_gb300 import (QLDPC_MSG_FP16, QLDPC_MSG_FP32, RelayConfig,  # noqa: E402
                                    RelayDecoder)

PREC = {QLDPC_MSG_FP32: "f32", QLDPC_MSG_FP16: "f16s"}


def _graph(rng, M, N, degrees, dc):
    """Random H with fault degrees drawn from `degrees` and check degrees at most dc (a fault
    that finds no room keeps fewer checks)."""
    H = np.zeros((M, N), dtype=np.uint8)
    for j in range(N):
        room = np.nonzero(H.sum(1) < dc)[0]
        d = min(int(rng.choice(degrees)), room.size)
        H[rng.choice(room, d, replace=False), j] = 1
    return H


# (checks, faults, fault degrees, check degree): whole warps of degree 2 and 3; a ragged last
# warp; degrees 0..4 mixed in every warp; sparse rows (many padding slots, empty rows);
# the 16- and 32-slot families with their 8 fault slots
GRAPHS = [(160, 384, (2, 3), 8), (161, 385, (3,), 8), (130, 301, (0, 1, 2, 3, 4), 8),
          (300, 320, (1, 2), 8), (120, 416, (2, 3), 16), (60, 351, (1, 2, 3, 5, 8), 32)]


@pytest.mark.parametrize("M,N,degrees,dc", GRAPHS)
@pytest.mark.parametrize("prec", [QLDPC_MSG_FP32, QLDPC_MSG_FP16])
@pytest.mark.parametrize("clip", [0.0, 12.0])
def test_random_graphs_match_the_mirror(M, N, degrees, dc, prec, clip):
    rng = np.random.default_rng(M * 1000 + N)
    H = _graph(rng, M, N, degrees, dc)
    p = rng.uniform(0.005, 0.08, N)
    P = DecodingProblem("random", H, np.zeros((1, N), np.uint8), p, {"code": "bb72"})
    sig = syndrome(P, (rng.random((150, N)) < p).astype(np.uint8))
    sig[:20] = rng.random((20, M)) < 0.5                   # mostly unsolvable: many legs
    gam = gamma_for(P, R=8, seed=N)
    cfg = dict(legs_after_first=8, iters_first=20, iters_later=15, stop_after_solutions=3)
    got = gpu_decode(P, gam, sig, RelayConfig(msg_precision=prec, llr_clip=clip, **cfg))
    prm = RelayParams(**cfg)
    if clip:
        prm.clip = clip
    ref = relay_decode(P.row_ptr, P.col_idx, P.p, gam, sig, prm, precision=PREC[prec])
    assert_same_decisions(got, ref, f"{M}x{N}/{PREC[prec]}/{clip}")


@pytest.mark.parametrize("prec", [QLDPC_MSG_FP32, QLDPC_MSG_FP16])
def test_recorded_messages_saturate_like_the_oracle(prec):
    """The passes hold fault-to-check messages unclamped; the trace records them clamped."""
    rng = np.random.default_rng(8)
    H = _graph(rng, 161, 385, (2, 3), 8)
    P = DecodingProblem("random", H, np.zeros((1, 385), np.uint8), rng.uniform(0.005, 0.08, 385),
                        {"code": "bb72"})
    sig = (rng.random((16, 161)) < 0.3).astype(np.uint8)
    gam = gamma_for(P, R=0)
    dec = RelayDecoder(P.row_ptr, P.col_idx, P.p, gam,
                       RelayConfig(legs_after_first=0, msg_precision=prec, llr_clip=12.0))
    marg, nu, mu = dec.trace_first_leg(torch.from_numpy(pack_bits(sig).view(np.int64)).cuda(), 12)
    torch.cuda.synchronize()
    dec.close()
    L, n, m = dmem_trace(P.row_ptr, P.col_idx, P.p, gam[0], sig, 12, precision=PREC[prec],
                         clip=12.0)
    assert np.abs(n).max() == 12.0
    for a, b in ((marg, L), (nu, n), (mu, m)):
        assert (a.cpu().numpy().transpose(1, 0, 2) == b).all()


# (code, rounds, shape the library takes): each compiled shape at a graph it is used for
SHAPES = [(BB72, 1, 64), (BB72, 4, 64), (BB72, 6, 64), (BB72, 7, 64), (BB72, 8, 128),
          (BB72, 10, 128), (BB72, 12, 128), (BB144, 8, 128), (BB144, 10, 128), (BB144, 11, 256),
          (BB144, 12, 256), (BB144, 13, 256), (BB144, 15, 256), (BB144, 18, 256),
          (BB144, 20, 256), (BB288, 12, 256), (BB288, 14, 256), (BB288, 15, 384),
          (BB288, 18, 256)]


@pytest.mark.parametrize("code,rounds,threads", SHAPES)
@pytest.mark.parametrize("prec", [QLDPC_MSG_FP32, QLDPC_MSG_FP16])
def test_library_shapes_match_the_mirror(code, rounds, threads, prec):
    """A batch above the small-batch shape's reach runs the narrow shape; its first shots are
    the oracle's, and the whole batch is the one a 1024-thread block decodes; a small batch
    (the wide shape) gives the same rows."""
    P = phenomenological_dem(code, rounds, 0.006)
    P.meta["code"] = "bb288" if code is BB288 else "bb144"
    n, few = 5000 if code is BB72 else 1300, 40
    sig = shots(P, n, rounds)[1]
    gam = gamma_for(P, R=40, seed=rounds)
    cfg = dict(legs_after_first=40, stop_after_solutions=3)
    got = gpu_decode(P, gam, sig, RelayConfig(msg_precision=prec, **cfg))
    assert got[4].block_threads == threads
    ref = relay_decode(P.row_ptr, P.col_idx, P.p, gam, sig[:few], RelayParams(**cfg),
                       precision=PREC[prec])
    assert_same_decisions(tuple(x[:few] for x in got[:4]), ref, "library's shape")
    wide = gpu_decode(P, gam, sig, RelayConfig(msg_precision=prec, block_threads=1024, **cfg))
    small = gpu_decode(P, gam, sig[:few], RelayConfig(msg_precision=prec, **cfg))
    for a, b, c in zip(got[:4], wide[:4], small[:4]):
        assert np.array_equal(a, b) and np.array_equal(a[:few], c)


def test_few_faults_with_many_checks_take_a_wide_enough_block():
    """90 faults and 1,200 checks: a 32-thread block would have more rows than a thread keeps
    syndrome bits for."""
    rng = np.random.default_rng(5)
    H = _graph(rng, 1200, 90, (2, 3, 4), 8)
    P = DecodingProblem("tall", H, np.zeros((1, 90), np.uint8), np.full(90, 0.05),
                        {"code": "bb72"})
    sig = syndrome(P, (rng.random((200, 90)) < 0.05).astype(np.uint8))
    gam = gamma_for(P, R=4, seed=2)
    cfg = dict(legs_after_first=4, stop_after_solutions=2)
    for prec in (QLDPC_MSG_FP32, QLDPC_MSG_FP16):
        got = gpu_decode(P, gam, sig, RelayConfig(msg_precision=prec, **cfg))
        ref = relay_decode(P.row_ptr, P.col_idx, P.p, gam, sig, RelayParams(**cfg),
                           precision=PREC[prec])
        assert_same_decisions(got, ref, f"tall/{PREC[prec]}")


def test_handles_that_share_a_shape_keep_their_shared_memory():
    """Two graphs on one compiled shape, the one with more shared memory created first."""
    big, small = (phenomenological_dem(BB288, t, 0.003) for t in (18, 16))
    for P in (big, small):
        P.meta["code"] = "bb288"
    cfg = RelayConfig(legs_after_first=20, stop_after_solutions=2)
    sig = shots(big, 800, 4)[1]
    gam = gamma_for(big, R=20)
    want = gpu_decode(big, gam, sig, cfg)
    first = RelayDecoder(big.row_ptr, big.col_idx, big.p, gam, cfg)
    second = RelayDecoder(small.row_ptr, small.col_idx, small.p, gamma_for(small, R=20), cfg)
    assert first.info.block_threads == second.info.block_threads
    assert first.info.smem_bytes > second.info.smem_bytes > 48 * 1024
    got = first.decode(torch.from_numpy(pack_bits(sig).view(np.int64)).cuda())
    torch.cuda.synchronize()
    for a, b in zip(got[1:], want[1:4]):                 # legs, converged, iterations
        assert np.array_equal(a.cpu().numpy(), b)
    first.close()
    second.close()
