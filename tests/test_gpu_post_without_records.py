"""Filtered-OSD on graphs with more than 64 KB of messages (no slot records in bytes) and on rows
with many padding slots: the kernel taken, and the oracle's result for every shot."""
import numpy as np
import pytest

from oracle.osd import OSDParams, bp_llrs, filtered_osd
from workloads import DecodingProblem, pack_bits, unpack_bits

from _cases import syndrome
from _launches import kernel_names

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
from paper_2511_21660_gb300 import FilteredOSD, QLDPC_OSD_SOLVED  # noqa: E402


def _problem(M, N, degrees, dc, seed):
    rng = np.random.default_rng(seed)
    H = np.zeros((M, N), dtype=np.uint8)
    H[0, :dc] = 1                                   # a full row: fixes the family
    rows = 1 + np.concatenate([rng.permutation(M - 1) for _ in range(4 * N // (M - 1) + 1)])
    k = 0
    for j in range(dc, N):
        d = int(rng.choice(degrees))
        H[rows[k:k + d], j] = 1
        k += d
    assert H.sum(1).max() == dc
    return DecodingProblem("rows", H, np.zeros((1, N), np.uint8), np.full(N, 0.02), {})


# (checks, faults, degrees, row slots, the kernel's threads and faults a thread)
CASES = [(2100, 1500, (2, 3), 8, "Li512ELi8E"), (1000, 1500, (2,), 8, "Li256ELi12E"),
         (40, 72, (2,), 8, "Li256ELi12E"), (1040, 900, (2, 3), 16, "Li512ELi8E")]


@pytest.mark.parametrize("M,N,degrees,dc,shape", CASES)
def test_osd_matches_oracle(M, N, degrees, dc, shape, tmp_path):
    P = _problem(M, N, degrees, dc, M + N)
    rng = np.random.default_rng(2)
    sig = syndrome(P, (rng.random((24, N)) < P.p).astype(np.uint8))
    prm = OSDParams(bp_iters=25, llr_confident=6.0, max_candidates=500)
    osd = FilteredOSD(P.row_ptr, P.col_idx, P.p, prm.bp_iters, prm.llr_confident,
                      prm.max_candidates)
    syn = torch.from_numpy(pack_bits(sig).view(np.int64)).cuda()
    cor = torch.zeros((24, osd.correction_words), dtype=torch.int64, device="cuda")
    names = kernel_names(lambda: osd.decode(syn, cor), tmp_path / "graph.dot", "osd_decode")
    assert len(names) == 1 and shape in names[0]
    cor.zero_()
    st, nc = (x.cpu().numpy() for x in osd.decode(syn, cor))
    got = unpack_bits(cor.cpu().numpy().view(np.uint64), N)
    osd.close()
    L = bp_llrs(P.row_ptr, P.col_idx, P.p, sig, prm.bp_iters, precision="f32")
    for b in range(24):
        c, s, n = filtered_osd(P.H, sig[b], L[b], prm)
        assert (st[b], nc[b]) == (s, n), b
        if s == QLDPC_OSD_SOLVED:
            assert np.array_equal(got[b], c), b
    assert (st == QLDPC_OSD_SOLVED).sum() >= 8
