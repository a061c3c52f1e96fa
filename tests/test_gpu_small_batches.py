"""The shape a batch runs by its size, and the narrow shapes themselves: batches above the
small-batch range, whose first shots are the oracle's and whose rows are a 1024-thread block's."""
import numpy as np
import pytest

from oracle.relay import RelayParams, relay_decode
from workloads import BB72, BB144, code_capacity_dem, pack_bits, phenomenological_dem

from _cases import assert_same_decisions, gamma_for, gpu_decode, shots
from _launches import kernel_names

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
from paper_2511_21660_gb300 import (QLDPC_MSG_FP16, QLDPC_MSG_FP32, RelayConfig,  # noqa: E402
                                    RelayDecoder, decode_mixed)

PREC = {QLDPC_MSG_FP32: "f32", QLDPC_MSG_FP16: "f16s"}
CFG = dict(legs_after_first=30, stop_after_solutions=3)


def _problem(code, rounds):
    P = code_capacity_dem(code, 0.05) if rounds == 0 else phenomenological_dem(code, rounds, 0.006)
    P.meta["code"] = "bb144"
    return P


# (code, rounds, {shots: threads and faults a thread}): the line is at 48 shots an SM for graphs of
# up to 1024 faults, at 4 for up to 3072
BATCHES = [(BB72, 0, {1: "Li64ELi4E", 7000: "Li64ELi4E", 9000: "Li32ELi3E"}),
           (BB144, 0, {1: "Li256ELi4E", 600: "Li256ELi4E", 7000: "Li256ELi4E",
                       9000: "Li64ELi4E"}),
           (BB72, 6, {1: "Li256ELi4E", 5000: "Li256ELi4E", 9000: "Li64ELi12E"}),
           (BB144, 12, {100: "Li512ELi6E", 2000: "Li256ELi11E"}),
           (BB144, 14, {1: "Li640ELi5E", 200: "Li640ELi5E", 2000: "Li640ELi5E"})]


@pytest.mark.parametrize("code,rounds,want", BATCHES)
def test_shape_by_batch_size(code, rounds, want, tmp_path):
    P = _problem(code, rounds)
    gam = gamma_for(P, R=0)
    dec = RelayDecoder(P.row_ptr, P.col_idx, P.p, gam, RelayConfig(legs_after_first=0))
    for n, shape in want.items():
        syn = torch.zeros((n, dec.syndrome_words), dtype=torch.int64, device="cuda")
        out = dec.outputs(n)
        names = kernel_names(lambda: dec.decode(syn, out=out), tmp_path / "graph.dot",
                             "fused_decode")
        assert len(names) == 1 and shape in names[0], (n, names)
    dec.close()


@pytest.mark.parametrize("pair,n,shape", [
    (((BB144, 12), (BB144, 14)), 200, "Li640ELi5E"), (((BB144, 12), (BB144, 14)), 2000, "Li640ELi5E"),
    (((BB72, 0), (BB144, 0)), 200, "Li256ELi4E"), (((BB72, 0), (BB144, 0)), 9000, "Li64ELi4E"),
    (((BB72, 6), (BB144, 12)), 2000, "Li512ELi6E")])
def test_shape_of_a_mixed_batch(pair, n, shape, tmp_path):
    probs = [_problem(c, r) for c, r in pair]
    gams = [gamma_for(P, R=6, seed=P.N) for P in probs]
    cfg = RelayConfig(legs_after_first=6, stop_after_solutions=2)
    decs = [RelayDecoder(P.row_ptr, P.col_idx, P.p, g, cfg) for P, g in zip(probs, gams)]
    code = np.arange(n) % 2
    stride = max(d.syndrome_words for d in decs)
    rows = np.zeros((n, stride), dtype=np.uint64)
    sigs = []
    for c, P in enumerate(probs):
        sigs.append(shots(P, int((code == c).sum()), 5)[1])
        w = pack_bits(sigs[c])
        rows[code == c, :w.shape[1]] = w
    codes = torch.from_numpy(code.astype(np.int32)).cuda()
    syn = torch.from_numpy(rows.view(np.int64)).cuda()
    names = kernel_names(lambda: decode_mixed(decs, codes, syn), tmp_path / "graph.dot",
                         "fused_decode_multi")
    assert len(names) == 1 and shape in names[0]
    got = [x.cpu().numpy() for x in decode_mixed(decs, codes, syn)]
    for c, (P, g) in enumerate(zip(probs, gams)):
        one = gpu_decode(P, g, sigs[c], cfg)
        for a, b in zip(got[1:], one[1:4]):
            assert np.array_equal(a[code == c], b)
    for d in decs:
        d.close()


@pytest.mark.parametrize("code,rounds,threads", [(BB72, 0, 32), (BB144, 0, 64), (BB72, 1, 64),
                                                 (BB72, 4, 64), (BB72, 6, 64), (BB72, 7, 64),
                                                 (BB72, 8, 128)])
@pytest.mark.parametrize("prec", [QLDPC_MSG_FP32, QLDPC_MSG_FP16])
def test_narrow_shapes_match_the_mirror(code, rounds, threads, prec):
    P = _problem(code, rounds)
    n, few = 9000, 40                            # above 48 shots an SM of 152
    sig = shots(P, n, rounds)[1]
    gam = gamma_for(P, R=30, seed=rounds)
    got = gpu_decode(P, gam, sig, RelayConfig(msg_precision=prec, **CFG))
    assert got[4].block_threads == threads and n > 48 * got[4].num_sms
    ref = relay_decode(P.row_ptr, P.col_idx, P.p, gam, sig[:few], RelayParams(**CFG),
                       precision=PREC[prec])
    assert_same_decisions(tuple(x[:few] for x in got[:4]), ref, "narrow shape")
    wide = gpu_decode(P, gam, sig, RelayConfig(msg_precision=prec, block_threads=1024, **CFG))
    small = gpu_decode(P, gam, sig[:few], RelayConfig(msg_precision=prec, **CFG))
    for a, b, c in zip(got[:4], wide[:4], small[:4]):
        assert np.array_equal(a, b) and np.array_equal(a[:few], c)
