"""Handles of two graphs on one kernel: the larger one, created first, still runs after the smaller
one has been created (post-processors, the plain kernel, the differentiable leg)."""
import numpy as np
import pytest

from workloads import BB144, BB288, pack_bits, phenomenological_dem

from _cases import gamma_for, shots

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
from paper_2511_21660_gb300 import (QLDPC_KERNEL_BASELINE, ClusterDecoder, FilteredOSD,  # noqa: E402
                                    RelayConfig, RelayDecoder, SoftDMem)


def _syndromes(P, n=40):
    F, sig = shots(P, n, 7)
    return [torch.from_numpy(pack_bits(x).view(np.int64)).cuda() for x in (sig, F)]


@pytest.mark.parametrize("make", [
    lambda P: FilteredOSD(P.row_ptr, P.col_idx, P.p, 25, 8.0, 500),
    lambda P: ClusterDecoder(P.row_ptr, P.col_idx, P.p, 25, -0.5, 4.5, 128, 512)],
    ids=["filtered-osd", "cluster"])
def test_post_processors(make):
    big, small = (phenomenological_dem(BB288, t, 0.01) for t in (18, 12))
    syn, _ = _syndromes(big)

    def run(h):
        cor = torch.zeros((syn.shape[0], h.correction_words), dtype=torch.int64, device="cuda")
        st, extra = h.decode(syn, cor)
        return [x.cpu().numpy() for x in (cor, st, extra)]
    first = make(big)
    want = run(first)
    second = make(small)
    for a, b in zip(run(first), want):
        assert np.array_equal(a, b)
    first.close()
    second.close()


def test_plain_kernel():
    big, small = (phenomenological_dem(BB144, t, 0.003) for t in (12, 9))
    syn, _ = _syndromes(big)
    cfg = RelayConfig(legs_after_first=5, kernel=QLDPC_KERNEL_BASELINE)
    first, second = (RelayDecoder(P.row_ptr, P.col_idx, P.p, gamma_for(problem, R=5), cfg)
                     for P, problem in ((big, _named(big)), (small, _named(small))))
    assert first.info.smem_bytes > second.info.smem_bytes > 48 * 1024
    iters = first.decode(syn)[3].cpu().numpy()
    assert (iters >= 1).all()
    first.close()
    second.close()


def _named(P):
    P.meta["code"] = "bb144"
    return P


def test_differentiable_leg():
    big, small = (phenomenological_dem(BB288, t, 0.01) for t in (18, 14))
    syn, flt = _syndromes(big, 4)
    first, second = (SoftDMem(P.row_ptr, P.col_idx, P.p, iterations=3, checkpoint_every=2)
                     for P in (big, small))

    def run(h, P, s, f):
        g = torch.full((P.N,), 0.1, device="cuda")
        a = torch.full((3,), 0.4, device="cuda")
        loss, _, ws = h.forward(s, f, g, a)
        return [x.cpu().numpy() for x in (loss, *h.backward(s, f, g, a, ws))]
    want = run(first, big, syn, flt)
    run(second, small, *_syndromes(small, 4))
    for a, b in zip(run(first, big, syn, flt), want):
        assert np.array_equal(a, b)
    first.close()
    second.close()
