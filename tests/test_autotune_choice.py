"""The autotuner's choice among the timed candidates (CPU), and that a tuned handle keeps the
small-batch shape when the library's own shape is the fastest (GPU)."""
import numpy as np
import pytest

from paper_2511_21660_gb300 import autotune

from _cases import gamma_for, problem, shots


def test_the_librarys_choice_is_a_candidate_and_wins_ties():
    assert 0 in autotune.CANDIDATES
    assert autotune.pick({"0/0": 1.01, "256/0": 1.0, "512/-1": 1.5}) == (0, 0)
    assert autotune.pick({"0/0": 1.2, "0/-1": 1.01, "256/0": 1.0}) == (0, -1)
    assert autotune.pick({"0/0": 1.2, "384/-1": 1.0}) == (384, -1)
    assert autotune.pick({"256/0": 1.0, "384/0": 0.9}) == (384, 0)


@pytest.mark.gpu
def test_a_tuned_handle_decodes_small_batches_with_the_wide_shape(tmp_path):
    torch = pytest.importorskip("torch")
    from paper_2511_21660_gb300 import RelayConfig, RelayDecoder
    from workloads import pack_bits

    from _launches import kernel_names
    P = problem("bb144_T12")
    gam = gamma_for(P, R=0)
    syn = torch.from_numpy(pack_bits(shots(P, 20000, 4)[1]).view(np.int64)).cuda()
    cfg = RelayConfig(legs_after_first=0)
    # the library's own block size named, against its choice: one shape on this batch
    (bt, _), ms = autotune.tune(P.row_ptr, P.col_idx, P.p, gam, cfg, syn, cache=None,
                                block_sizes=(0, 1024), tail_options=(0,))
    assert set(ms) == {"0/0", "1024/0"}
    assert bt == 0 or ms["1024/0"] < ms["0/0"]
    cfg.block_threads = 0
    dec = RelayDecoder(P.row_ptr, P.col_idx, P.p, gam, cfg)
    few = syn[:100].contiguous()
    names = kernel_names(lambda: dec.decode(few), tmp_path / "graph.dot", "fused_decode")
    assert len(names) == 1 and "Li512ELi6E" in names[0]
    dec.close()
