"""Which resuming launches a batch queues: a split launch always where the graph has one, and
beside it the one-block launch unless the batch has too few shots to give every cluster more than
one record.  A small batch can consist of unsolvable syndromes alone, so the number of its shots
is the only bound on its records that the host knows."""
import ctypes
import re

import numpy as np
import pytest

from workloads import BB72, BB144, BB288, pack_bits, phenomenological_dem

from _cases import gamma_for, gpu_decode

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
from paper_2511_21660_gb300 import (QLDPC_MSG_FP16, QLDPC_MSG_FP32, RelayConfig,  # noqa: E402
                                    RelayDecoder, decode_grouped)


def _problem(code, rounds):
    P = phenomenological_dem(code, rounds, 0.02)
    P.meta["code"] = "bb288" if code is BB288 else "bb144"
    return P


def _unsolvable(P, n):
    """Random syndromes: nearly all of them outlast the first leg and the later ones."""
    return (np.random.default_rng(n).random((n, P.M)) < 0.5).astype(np.uint8)


def _decoder(P, prec=QLDPC_MSG_FP32, **cfg):
    return RelayDecoder(P.row_ptr, P.col_idx, P.p, gamma_for(P, R=cfg["legs_after_first"]),
                        RelayConfig(msg_precision=prec, **cfg))


def _queued(call, tmp_path):
    """(split launches, one-block resuming launches) among the kernels that `call` queues: the
    kernel nodes of its captured graph, as the driver prints them."""
    call()                                       # first-use work happens outside the capture
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph):
        call()
    path = str(tmp_path / "graph.dot")
    driver = ctypes.CDLL("libcuda.so.1")
    assert driver.cuGraphDebugDotPrint(ctypes.c_void_p(graph.raw_cuda_graph()), path.encode(),
                                       ctypes.c_uint(0)) == 0
    # mangled names; the last template argument of fused_decode is its RESUME flag
    names = re.findall(r"\w*(?:split_resume|fused_decode)\w*", open(path).read())
    assert any("fused_decode" in n for n in names)
    return (sum("split_resume" in n for n in names),
            sum("fused_decode" in n and "Lb1E" in n for n in names))


CFG = dict(legs_after_first=4, iters_first=10, iters_later=10, tail_cut_iters=1)


@pytest.mark.parametrize("code,rounds", [(BB72, 7), (BB144, 12), (BB288, 18)])
@pytest.mark.parametrize("prec", [QLDPC_MSG_FP32, QLDPC_MSG_FP16])
def test_launches_by_batch_size(code, rounds, prec, tmp_path):
    P = _problem(code, rounds)
    dec = _decoder(P, prec, **CFG)
    many = 2 * dec.info.num_sms + 1              # above 4 blocks a cluster, 8 of 256 threads an SM
    sig = _unsolvable(P, 8 * many)
    syn = torch.from_numpy(pack_bits(sig).view(np.int64)).cuda()
    for n, want in ((1, (1, 0)), (many, (1, 1)), (8 * many, (1, 1))):
        s = syn[:n].contiguous()
        out = dec.outputs(n)
        assert _queued(lambda: dec.decode(s, out=out), tmp_path) == want, n
    dec.close()


def test_grouped_call_queues_both(tmp_path):
    P = _problem(BB144, 12)
    decs = [_decoder(P, **CFG), _decoder(_problem(BB72, 7), **CFG)]
    n = 2 * decs[0].info.num_sms + 1
    codes = torch.zeros(n, dtype=torch.int32, device="cuda")
    codes[::2] = 1
    syn = torch.zeros((n, decs[0].syndrome_words), dtype=torch.int64, device="cuda")
    assert _queued(lambda: decode_grouped(decs, codes, syn), tmp_path) == (2, 2)
    for d in decs:
        d.close()


@pytest.mark.parametrize("n", [40, 150, 300])
def test_unsolvable_batches_match_the_single_launch(n):
    P = _problem(BB144, 12)
    sig = _unsolvable(P, n)
    gam = gamma_for(P, R=4)
    on = gpu_decode(P, gam, sig, RelayConfig(**CFG))
    off = gpu_decode(P, gam, sig, RelayConfig(**dict(CFG, tail_cut_iters=-1)))
    assert (on[1] > 1).sum() > n // 2            # more than half went through a second launch
    for a, b in zip(on[:4], off[:4]):
        assert np.array_equal(a, b)
