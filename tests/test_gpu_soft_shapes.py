"""The forward kernel of the differentiable leg by the size of the graph's state, and a graph that
runs the wide blocks against the FP64 oracle (with the tolerances of the 12-round gross graph)."""
import numpy as np
import pytest

from oracle.soft import soft_dmem
from workloads import BB72, BB144, BB288, pack_bits, phenomenological_dem, sample_faults, \
    syndromes_of

from _launches import kernel_names

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
from paper_2511_21660_gb300 import SoftDMem  # noqa: E402


def _inputs(P, B, T, seed):
    F = sample_faults(P.p, seed, B)
    s = syndromes_of(P.row_ptr, P.col_idx, F)
    rng = np.random.default_rng(seed)
    gam = rng.uniform(0.0, 0.3, P.N).astype(np.float32)
    alpha = rng.uniform(0.25, 0.4, T).astype(np.float32)
    dev = [torch.from_numpy(pack_bits(x).view(np.int64)).cuda() for x in (s, F)]
    return F, s, gam, alpha, dev + [torch.from_numpy(x).cuda() for x in (gam, alpha)]


# five blocks of 40 and 43 KB of state fit an SM, of 53 KB and more do not
@pytest.mark.parametrize("code,rounds,threads", [(BB72, 6, 320), (BB144, 12, 320),
                                                 (BB144, 13, 320), (BB144, 16, 512),
                                                 (BB288, 18, 512)])
def test_forward_threads_by_state_size(code, rounds, threads, tmp_path):
    P = phenomenological_dem(code, rounds, 0.003)
    soft = SoftDMem(P.row_ptr, P.col_idx, P.p, iterations=3, checkpoint_every=3)
    *_, dev = _inputs(P, 2, 3, 5)
    names = kernel_names(lambda: soft.forward(*dev), tmp_path / "graph.dot", "soft_forward")
    assert len(names) == 1 and f"Li8ELi{threads}E" in names[0]
    soft.close()


def test_wide_blocks_track_the_fp64_oracle():
    P = phenomenological_dem(BB144, 16, 0.003)
    F, s, gam, alpha, dev = _inputs(P, 6, 25, 29)
    L_ref, gg_ref, ga_ref, m_ref = soft_dmem(P.row_ptr, P.col_idx, P.p, gam.astype(np.float64),
                                             alpha.astype(np.float64), s, F, eps=2.0 ** -23,
                                             marginals=True)
    soft = SoftDMem(P.row_ptr, P.col_idx, P.p, iterations=25, checkpoint_every=5)
    loss, marg, ws = soft.forward(*dev, marginals=True)
    gg, ga = soft.backward(*dev, ws)
    torch.cuda.synchronize()
    err = np.abs(marg.cpu().numpy() - m_ref) / np.maximum(1.0, np.abs(m_ref))
    assert err.max() <= 1e-3, err.max()
    assert abs(loss.item() - L_ref) <= 1e-4 * L_ref
    assert np.abs(gg.cpu().numpy() - gg_ref).max() <= 1e-3 * np.abs(gg_ref).max()
    assert np.abs(ga.cpu().numpy() - ga_ref).max() <= 1e-3 * np.abs(ga_ref).max()
    soft.close()
