"""GPU parity of full-entity scoring: top-k ids bit-exact against the fp32 oracle (both
sides decide the order in fp32 with the same per-pair operation order), scores at 1e-4,
ranks exact, MRR within 1e-3; exact ties, k > |E|, the list-overflow path."""
import numpy as np
import pytest

from parity_util import GpuSide, Problem, assert_close

pytestmark = pytest.mark.gpu


def _infer(gpu, qh, qr, tt, K):
    t = gpu.torch
    dev = gpu.ent.device
    nq = len(qh)
    ids = t.empty((nq, K), dtype=t.int32, device=dev); sc = t.empty((nq, K), dtype=t.float32, device=dev)
    ranks = t.empty(nq, dtype=t.int32, device=dev)
    gpu.kge.score_all_topk(gpu.dev_i32(qh), gpu.dev_i32(qr), K, gpu.dev_i32(tt), ids, sc, ranks)
    assert gpu.kge.get_status() == 0
    return ids.cpu().numpy(), sc.cpu().numpy(), ranks.cpu().numpy()


@pytest.mark.parametrize("score,p", [("transe", 1), ("transe", 2), ("distmult", 1), ("complex", 1),
                                     ("transh", 1), ("transh", 2), ("rotate", 2), ("rotate", 1), ("rotate_real_l1", 1)])
def test_topk_rank_mrr_against_fp32_oracle(oracle32, oracle64, score, p):
    import kge_synth
    E, R, d, K, nq = 5000, 9, 40, 10, 70          # chunks 1024 and 3976; ragged tiles
    prob = Problem(E=E, R=R, T=100, d=d, score=score, p_norm=p, B=4, N=4, P=1, graph_seed=11)
    prob.ent[3000] = prob.ent[17]; prob.ent[4999] = prob.ent[17]; prob.ent[1] = prob.ent[0]   # exact ties
    qh, qr, tt = kge_synth.make_queries(E, R, nq, seed=11)
    tt[0] = qh[0]; tt[1] = 4999; tt[2] = 17
    gpu = GpuSide(prob, max_queries=nq, topk=K, load_graph=False)
    ids, sc, ranks = _infer(gpu, qh, qr, tt, K)
    cfg = prob.oracle_cfg()
    o_ids, o_sc, o_ranks = oracle32.score_all_topk(cfg, prob.ent, prob.rel, prob.relw, qh, qr, K, true_tails=tt)
    if score in ("rotate", "rotate_real_l1"):
        # sin / cos come from different math libraries: compare as sets, audit near-ties
        r_ids, r_sc, r_ranks = oracle64.score_all_topk(cfg, prob.ent, prob.rel, prob.relw, qh, qr, K + 5, true_tails=tt)
        for q in range(nq):
            extra = set(ids[q]) - set(r_ids[q, :K])
            for e in extra:
                assert e in set(r_ids[q]), "id outside the oracle's top (k+5)"
                f = r_sc[q][list(r_ids[q]).index(e)]
                assert abs(f - r_sc[q, K - 1]) <= 1e-4 * abs(f)
        assert_close(sc, r_sc[:, :K], what="scores")
        assert np.abs(ranks - r_ranks).max() <= 2
    else:
        assert (ids == o_ids).all()
        assert (sc == o_sc).all() or np.allclose(sc, o_sc, rtol=1e-6)
        assert (ranks == o_ranks).all()
    mrr = gpu.kge.eval_mrr(gpu.dev_i32(qh), gpu.dev_i32(qr), gpu.dev_i32(tt), 10)
    assert abs(mrr - oracle64.mrr(o_ranks, 10)) <= 1e-3
    mrr0 = gpu.kge.eval_mrr(gpu.dev_i32(qh), gpu.dev_i32(qr), gpu.dev_i32(tt), 0)
    assert abs(mrr0 - oracle64.mrr(o_ranks, 0)) <= 1e-3
    # the same metric from ranks the caller already holds (no second pass over the table)
    ranks_dev = gpu.dev_i32(ranks)
    assert gpu.kge.mrr_from_ranks(ranks_dev, 10) == mrr and gpu.kge.mrr_from_ranks(ranks_dev, 0) == mrr0
    if score not in ("rotate", "rotate_real_l1"):
        assert abs(mrr - oracle64.mrr(o_ranks, 10)) <= 1e-12 and abs(mrr0 - oracle64.mrr(o_ranks, 0)) <= 1e-12


@pytest.mark.parametrize("score,p,d", [("transe", 1, 128), ("distmult", 1, 40), ("transe", 2, 64), ("complex", 1, 128)])
def test_five_query_tiles_with_a_ragged_last_one(oracle32, score, p, d):
    """300 queries (a ragged fifth 64-query tile) against 3,000 entities (ragged last tile, chunks 1024 + 1976)
    with exact ties: ids, scores and ranks bit-exact against the fp32 oracle."""
    import kge_synth
    E, R, K, nq = 3000, 9, 10, 300
    prob = Problem(E=E, R=R, T=100, d=d, score=score, p_norm=p, B=4, N=4, P=1, graph_seed=19)
    prob.ent[2900] = prob.ent[17]; prob.ent[1] = prob.ent[0]
    qh, qr, tt = kge_synth.make_queries(E, R, nq, seed=19)
    tt[0] = qh[0]; tt[1] = 2900; tt[2] = 17
    gpu = GpuSide(prob, max_queries=nq, topk=K, load_graph=False)
    ids, sc, ranks = _infer(gpu, qh, qr, tt, K)
    o_ids, o_sc, o_ranks = oracle32.score_all_topk(prob.oracle_cfg(), prob.ent, prob.rel, prob.relw, qh, qr, K, true_tails=tt)
    assert (ids == o_ids).all() and (ranks == o_ranks).all()
    assert (sc == o_sc).all() or np.allclose(sc, o_sc, rtol=1e-6)


@pytest.mark.parametrize("score,E,d", [("distmult", 5000, 64), ("complex", 5000, 64), ("distmult", 70000, 128),
                                       ("complex", 40000, 256)])
def test_tensor_core_topk_against_bf16_operand_oracle(oracle64, score, E, d):
    """Full-entity scoring on tensor cores (bf16 operands, fp32 accumulation) against the oracle
    with bf16-rounded operands.  The accumulation order differs, so the lists are compared as
    sets with a near-tie audit (2e-2 relative is the stated bound of this path; 1e-4 is used),
    ranks within 2, MRR within 1e-3.  E = 5000 leaves ragged 256-entity tiles, nq = 200 two query tiles, one per
    CTA until a chunk has 148 entity tiles: the later chunks at E = 70,000 pass two by one entity tile at d = 128 (two
    slices of the ring), those at d = 256 one (four)."""
    import kge_synth
    R, K, nq = 9, 10, 200
    prob = Problem(E=E, R=R, T=100, d=d, score=score, p_norm=1, B=8, N=8, P=1, graph_seed=12, tc=True)
    qh, qr, tt = kge_synth.make_queries(E, R, nq, seed=12)
    tt[0] = qh[0]
    gpu = GpuSide(prob, max_queries=nq, topk=K, load_graph=False)
    ids, sc, ranks = _infer(gpu, qh, qr, tt, K)
    cfg = prob.oracle_cfg()
    r_ids, r_sc, r_ranks = oracle64.score_all_topk(cfg, prob.ent, prob.rel, prob.relw, qh, qr, K + 5, true_tails=tt)
    for q in range(nq):
        assert len(set(ids[q])) == K
        for e in set(ids[q]) - set(r_ids[q, :K]):
            assert e in set(r_ids[q]), "id outside the oracle's top (k+5)"
            f = r_sc[q][list(r_ids[q]).index(e)]
            assert abs(f - r_sc[q, K - 1]) <= 1e-4 * abs(f) + 1e-6
    assert_close(sc, r_sc[:, :K], atol=1e-5, what="scores")
    assert np.abs(ranks - r_ranks).max() <= 2
    mrr = gpu.kge.eval_mrr(gpu.dev_i32(qh), gpu.dev_i32(qr), gpu.dev_i32(tt), 0)
    assert abs(mrr - oracle64.mrr(r_ranks, 0)) <= 1e-3


def test_config1_mrr_after_training(oracle32, oracle64):
    """The small configuration: 10 SGD steps, then MRR of the first 100 triples ranked against
    all 1,000 entities.  Inference parity is taken on the GPU's own trained tables."""
    prob = Problem(E=1000, R=10, T=20000, d=32, score="distmult", loss="logsigmoid", B=64, N=128, P=2,
                   lr=0.1, seed=0, graph_seed=0)
    gpu = GpuSide(prob, max_queries=100, topk=10)
    for step in range(10):
        gpu.kge.train_step(step, prob.lr)
    qh, qr, tt = prob.h[:100], prob.r[:100], prob.t[:100]
    ids, sc, ranks = _infer(gpu, qh, qr, tt, 10)
    ent, rel, _ = gpu.tables()
    o_ids, o_sc, o_ranks = oracle32.score_all_topk(prob.oracle_cfg(), ent, rel, None, qh, qr, 10, true_tails=tt)
    assert (ids == o_ids).all() and (ranks == o_ranks).all()
    assert abs(gpu.kge.eval_mrr(gpu.dev_i32(qh), gpu.dev_i32(qr), gpu.dev_i32(tt), 0) - oracle64.mrr(o_ranks, 0)) <= 1e-3


def test_k_larger_than_entities_and_single_query(oracle32):
    prob = Problem(E=9, R=2, T=50, d=16, score="transe", p_norm=1, B=4, N=4, P=1, graph_seed=12)
    gpu = GpuSide(prob, max_queries=4, topk=12, load_graph=False)
    ids, sc, ranks = _infer(gpu, np.array([3]), np.array([1]), np.array([4]), 12)
    o_ids, o_sc, o_ranks = oracle32.score_all_topk(prob.oracle_cfg(), prob.ent, prob.rel, None, [3], [1], 12, true_tails=[4])
    assert (ids == o_ids).all() and (ranks == o_ranks).all()
    assert (ids[0, 9:] == -1).all() and np.isneginf(sc[0, 9:]).all()


def test_empty_query_batch_is_a_no_op(oracle32):
    """nq = 0: the call returns success, launches nothing and leaves the outputs alone."""
    prob = Problem(E=9, R=2, T=50, d=16, score="transe", p_norm=1, B=4, N=4, P=1, graph_seed=12)
    gpu = GpuSide(prob, max_queries=4, topk=3, load_graph=False)
    t = gpu.torch
    dev = gpu.ent.device
    ids = t.full((1, 3), 77, dtype=t.int32, device=dev); sc = t.full((1, 3), 5.0, dtype=t.float32, device=dev)
    empty = t.empty(0, dtype=t.int32, device=dev)
    before = gpu.kge.launch_count()
    gpu.kge.score_all_topk(empty, empty, 3, None, ids, sc, None)
    assert gpu.kge.get_status() == 0 and gpu.kge.launch_count() == before
    assert (ids.cpu().numpy() == 77).all() and (sc.cpu().numpy() == 5.0).all()


def test_rising_scores_take_the_overflow_path(oracle32):
    """Scores that grow with the entity id make every entity of a chunk beat the current
    k-th best, which fills the candidate list; the library must redo the chunk in pieces."""
    E, d, K = 6000, 16, 5
    prob = Problem(E=E, R=2, T=50, d=d, score="distmult", B=4, N=4, P=1, graph_seed=13)
    prob.ent[:] = 0.0
    prob.ent[:, 0] = np.arange(E, dtype=np.float32) / E + 0.5
    prob.rel[:] = 1.0
    gpu = GpuSide(prob, max_queries=8, topk=K, load_graph=False)
    qh, qr, tt = np.array([10, 4000, 5999]), np.array([0, 1, 0]), np.array([0, 5999, 3000])
    ids, sc, ranks = _infer(gpu, qh, qr, tt, K)
    o_ids, _, o_ranks = oracle32.score_all_topk(prob.oracle_cfg(), prob.ent, prob.rel, None, qh, qr, K, true_tails=tt)
    assert (ids == o_ids).all() and (ranks == o_ranks).all()
    assert (ids[0] == np.arange(E - 1, E - 1 - K, -1)).all()


@pytest.mark.parametrize("d", [28, 32, 36, 64, 68, 96, 132, 196, 260])
@pytest.mark.parametrize("score,p,K", [("transe", 1, 10), ("transe", 2, 100), ("distmult", 1, 129)])
def test_row_widths_at_the_edges_of_a_staged_box(oracle32, score, p, d, K):
    """Rows that end at, before and after the 32-float boxes and 64-float stages of the score tile; lists of up to 128 places
    (cut down before they are sorted) and one more; 65 queries (a second tile of one row), 2,500 entities in two chunks (K = 129: three)."""
    import kge_synth
    E, R, nq = 2500, 5, 65
    prob = Problem(E=E, R=R, T=100, d=d, score=score, p_norm=p, B=4, N=4, P=1, graph_seed=31)
    prob.ent[2400] = prob.ent[17]; prob.ent[1000] = prob.ent[17]
    qh, qr, tt = kge_synth.make_queries(E, R, nq, seed=31)
    tt[0] = qh[0]; tt[1] = 2400; qh[2] = 17
    gpu = GpuSide(prob, max_queries=nq, topk=K, load_graph=False)
    ids, sc, ranks = _infer(gpu, qh, qr, tt, K)
    o_ids, o_sc, o_ranks = oracle32.score_all_topk(prob.oracle_cfg(), prob.ent, prob.rel, None, qh, qr, K, true_tails=tt)
    assert (ids == o_ids).all() and (ranks == o_ranks).all()
    assert (sc == o_sc).all()


@pytest.mark.parametrize("score,tc,d", [("distmult", False, 32), ("distmult", True, 64), ("distmult", False, 16)])
@pytest.mark.parametrize("lo,hi", [(3000, 9000), (1024, 30000)])
@pytest.mark.parametrize("K", [1, 40])
def test_scores_that_rise_along_a_stretch(oracle32, score, tc, d, lo, hi, K):
    """A list that fills up in the middle of the table: the chunk is redone in pieces (of several sizes in the longer
    stretch) while the chunks queued behind it wait.  Values with eight significant bits: exact in every arithmetic, with
    ties decided by the id."""
    E = 40_000
    prob = Problem(E=E, R=2, T=50, d=d, score=score, B=4, N=4, P=1, graph_seed=13, tc=tc)
    prob.ent[:] = 0.0
    prob.ent[:, 0] = 0.25
    prob.ent[lo:hi, 0] = 0.5 + np.floor(np.arange(hi - lo) * 127.0 / (hi - lo)) / 256.0
    prob.rel[:] = 1.0
    gpu = GpuSide(prob, max_queries=70, topk=K, load_graph=False)
    rng = np.random.default_rng(5)
    qh, qr, tt = rng.integers(0, E, 66), rng.integers(0, 2, 66), rng.integers(0, E, 66)
    ids, sc, ranks = _infer(gpu, qh, qr, tt, K)
    o_ids, o_sc, o_ranks = oracle32.score_all_topk(prob.oracle_cfg(), prob.ent, prob.rel, None, qh, qr, K, true_tails=tt)
    assert (ids == o_ids).all() and (ranks == o_ranks).all() and (sc == o_sc).all()


@pytest.mark.parametrize("score,p,d", [("transe", 1, 40), ("transe", 2, 96), ("distmult", 1, 132), ("complex", 1, 28), ("transh", 1, 40), ("transh", 2, 36)])
@pytest.mark.parametrize("K", [10, 100])
def test_several_filtered_chunks(oracle32, score, p, d, K):
    """17,000 entities: chunks of 1,024, then four (K = 100: two) times what went before, so that the running lists are merged,
    and the thresholds tightened, at least twice after the first selection."""
    import kge_synth
    E, R, nq = 17_000, 5, 66
    prob = Problem(E=E, R=R, T=100, d=d, score=score, p_norm=p, B=4, N=4, P=1, graph_seed=33)
    prob.ent[16_990] = prob.ent[17]; prob.ent[6000] = prob.ent[17]
    qh, qr, tt = kge_synth.make_queries(E, R, nq, seed=33)
    tt[0] = qh[0]; tt[1] = 16_990; qh[2] = 17
    gpu = GpuSide(prob, max_queries=nq, topk=K, load_graph=False)
    ids, sc, ranks = _infer(gpu, qh, qr, tt, K)
    o_ids, o_sc, o_ranks = oracle32.score_all_topk(prob.oracle_cfg(), prob.ent, prob.rel, prob.relw, qh, qr, K, true_tails=tt)
    assert (ids == o_ids).all() and (ranks == o_ranks).all()
    assert (sc == o_sc).all() or np.allclose(sc, o_sc, rtol=1e-6)


@pytest.mark.parametrize("score,d", [("transe", 16), ("transe", 84), ("transh", 36)])
@pytest.mark.parametrize("nq", [1, 63, 64, 65])
def test_ranks_of_few_queries(oracle32, score, d, nq):
    """Rank counts of a tile's rows, whole and ragged, in every tile kernel; without true tails nothing is counted."""
    import kge_synth
    E, R, K = 1500, 5, 3
    prob = Problem(E=E, R=R, T=100, d=d, score=score, p_norm=1, B=4, N=4, P=1, graph_seed=35)
    qh, qr, tt = kge_synth.make_queries(E, R, nq, seed=35)
    tt[0] = E - 1
    gpu = GpuSide(prob, max_queries=nq, topk=K, load_graph=False)
    ids, sc, ranks = _infer(gpu, qh, qr, tt, K)
    o_ids, o_sc, o_ranks = oracle32.score_all_topk(prob.oracle_cfg(), prob.ent, prob.rel, prob.relw, qh, qr, K, true_tails=tt)
    assert (ids == o_ids).all() and (ranks == o_ranks).all()
    t = gpu.torch
    ids2, sc2 = t.empty((nq, K), dtype=t.int32, device=gpu.ent.device), t.empty((nq, K), dtype=t.float32, device=gpu.ent.device)
    gpu.kge.score_all_topk(gpu.dev_i32(qh), gpu.dev_i32(qr), K, None, ids2, sc2)
    assert (ids2.cpu().numpy() == ids).all() and (sc2.cpu().numpy() == sc).all()


@pytest.mark.parametrize("score,tc,d", [("transe", False, 64), ("transh", False, 32), ("distmult", False, 16), ("distmult", True, 64)])
def test_a_rise_after_a_restart(oracle32, score, tc, d):
    """Two stretches of rising scores: the chunks that were cut down in the first have grown again when the second fills the
    lists, and the second begins inside a chunk of a few queued ones."""
    E, K = 150_000, 7
    prob = Problem(E=E, R=2, T=50, d=d, score=score, p_norm=1, B=4, N=4, P=1, graph_seed=13, tc=tc)
    step = np.zeros(E, np.float32)
    step[2000:5000] = 0.25 + np.arange(3000, dtype=np.float32) // 24 / 512.0          # up to 0.494
    step[90_000:130_000] = 0.5 + np.arange(40_000, dtype=np.float32) // 160 / 512.0   # up to 0.986
    prob.ent[:] = 0.0
    if score == "distmult":
        prob.ent[:, 0] = 0.25 + step.astype(np.float32) if not tc else np.round((0.25 + step) * 128) / 128
        prob.rel[:] = 1.0
    else:
        prob.ent[:, 0] = step                             # distance to the query's 2 (a head of 0 and a relation of 2) falls along the stretch
        prob.rel[:] = 0.0; prob.rel[:, 0] = 2.0
        if prob.relw is not None:
            prob.relw[:] = 0.0; prob.relw[:, 1] = 1.0
    gpu = GpuSide(prob, max_queries=70, topk=K, load_graph=False)
    rng = np.random.default_rng(5)
    qh, qr, tt = rng.integers(0, 1500, 66), rng.integers(0, 2, 66), rng.integers(0, E, 66)
    ids, sc, ranks = _infer(gpu, qh, qr, tt, K)
    o_ids, o_sc, o_ranks = oracle32.score_all_topk(prob.oracle_cfg(), prob.ent, prob.rel, prob.relw, qh, qr, K, true_tails=tt)
    assert (ids == o_ids).all() and (ranks == o_ranks).all() and (sc == o_sc).all()


# tensor cores: one, two and three tiles of 128 queries, a table that ends inside and at the end of a 256-entity tile, CTAs of their own
# for every query group, lists that take many candidates
@pytest.mark.parametrize("nq,E,d,K", [(1, 3001, 64, 10), (128, 4352, 128, 40), (129, 6000, 128, 1), (257, 9000, 64, 100), (385, 6001, 192, 10), (130, 20000, 384, 40),
                                      (2900, 5000, 64, 10), (300, 1500, 512, 5)])
def test_tensor_core_query_groups(oracle64, nq, E, d, K):
    import kge_synth
    prob = Problem(E=E, R=9, T=100, d=d, score="distmult", B=8, N=8, P=1, graph_seed=47, tc=True)
    qh, qr, tt = kge_synth.make_queries(E, 9, nq, seed=47)
    gpu = GpuSide(prob, max_queries=nq, topk=K, load_graph=False)
    ids, sc, ranks = _infer(gpu, qh, qr, tt, K)
    r_ids, r_sc, r_ranks = oracle64.score_all_topk(prob.oracle_cfg(), prob.ent, prob.rel, prob.relw, qh, qr, K + 5, true_tails=tt)
    for q in range(nq):
        assert len(set(ids[q])) == K
        for e in set(ids[q]) - set(r_ids[q, :K]):          # (near ties only: the sums' order differs)
            assert e in set(r_ids[q])
            f = r_sc[q][list(r_ids[q]).index(e)]
            assert abs(f - r_sc[q, K - 1]) <= 1e-4 * abs(f) + 1e-6
    assert_close(sc, r_sc[:, :K], atol=1e-5, what="scores")
    assert np.abs(ranks - r_ranks).max() <= 2
    t = gpu.torch                                          # without true tails: the same lists
    ids2 = t.empty((nq, K), dtype=t.int32, device=gpu.ent.device); sc2 = t.empty((nq, K), dtype=t.float32, device=gpu.ent.device)
    gpu.kge.score_all_topk(gpu.dev_i32(qh), gpu.dev_i32(qr), K, None, ids2, sc2)
    assert (ids2.cpu().numpy() == ids).all() and (sc2.cpu().numpy() == sc).all()


def test_tensor_core_lists_of_equal_scores(oracle64):
    """Every entity the same row: all scores of a query are equal, and the smallest ids win without filling a candidate list."""
    import kge_synth
    E, nq, K = 40000, 140, 10
    prob = Problem(E=E, R=9, T=100, d=64, score="distmult", B=8, N=8, P=1, graph_seed=49, tc=True)
    prob.ent[:] = prob.ent[0]
    qh, qr, tt = kge_synth.make_queries(E, 9, nq, seed=49)
    gpu = GpuSide(prob, max_queries=nq, topk=K, load_graph=False)
    ids, _, _ = _infer(gpu, qh, qr, tt, K)
    assert (ids == np.arange(K)).all()


@pytest.mark.parametrize("d,E", [(64, 9000), (64, 120_000), (192, 9000)])        # (120,000: two query tiles per CTA)
def test_tensor_core_queries_outside_the_call_score_infinity(d, E):
    """A call with fewer queries than the workspace holds, where the rest of the query vectors' memory makes every score +inf and the
    rest of the thresholds' ids lie beyond the table: nothing of it reaches the call, which ends and gives what a call with as
    many queries as the workspace holds gives."""
    import kge_synth
    R, K, nq, most = 5, 10, 130, 400
    prob = Problem(E=E, R=R, T=100, d=d, score="distmult", B=8, N=8, P=1, graph_seed=51, tc=True)
    prob.ent = np.abs(prob.ent)                                # (no +inf - inf among the sums)
    qh, qr, tt = kge_synth.make_queries(E, R, nq, seed=51)
    gpu = GpuSide(prob, max_queries=nq, topk=K, load_graph=False)
    want = _infer(gpu, qh, qr, tt, K)
    t = gpu.torch
    need = gpu.kge.workspace_bytes(0, most, K)
    space = t.full((need + 512,), 0x7F, dtype=t.uint8, device=gpu.ent.device)
    space[::2] = 0x80                                          # 0x7F80: +inf as bf16, 0x7F807F80 as an id
    gpu.kge.bind(gpu.ent, gpu.rel, None, max_queries=most, topk=K, workspace=space[(-space.data_ptr()) % 256:][:need])
    for got, exact in zip(_infer(gpu, qh, qr, tt, K), want):
        assert (got == exact).all()


# an odd number of query tiles where two share a CTA, for which the last group has one; as many queries as the workspace holds, so
# that what lies behind the lists is the workspace's next array
@pytest.mark.parametrize("nq,d", [(300, 128), (128, 64), (290, 192)])
def test_tensor_core_scoring_after_waits_that_run_out(nq, d):
    """Limits so short that a wait runs out anywhere in the scoring: the call reports KGE_ERR_TIMEOUT (or got by), and the next
    one, which uses the same copy of the table, gives what it gave before."""
    import kge_synth
    E, R, K = 60_000, 5, 10
    prob = Problem(E=E, R=R, T=100, d=d, score="distmult", B=8, N=8, P=1, graph_seed=53, tc=True)
    qh, qr, tt = kge_synth.make_queries(E, R, nq, seed=53)
    gpu = GpuSide(prob, max_queries=nq, topk=K, load_graph=False)
    want = _infer(gpu, qh, qr, tt, K)
    t = gpu.torch
    out = [t.empty((nq, K), dtype=t.int32, device=gpu.ent.device), t.empty((nq, K), device=gpu.ent.device), t.empty(nq, dtype=t.int32, device=gpu.ent.device)]
    ran_out = 0
    for tries in (1, 1, 1, 1, 2, 4, 8, 16, 64):
        gpu.kge.debug_set_wait_limit(tries)
        gpu.kge.score_all_topk(gpu.dev_i32(qh), gpu.dev_i32(qr), K, gpu.dev_i32(tt), *out)
        status = gpu.kge.get_status()
        assert status in (0, -11)
        ran_out += status != 0
    assert ran_out
    gpu.kge.debug_set_wait_limit(0)
    for got, exact in zip(_infer(gpu, qh, qr, tt, K), want):
        assert (got == exact).all()


def _shared_groups():
    """The fewest query groups (from nine on) that leave so many SMs idle with CTAs of their own that all CTAs share them."""
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    return next(g for g in range(9, sms) if sms // g * g * 16 < sms * 15)


# tensor cores, groups of queries that share the CTAs: a CTA crosses from one group to the next, loads its queries and hands the ones
# before over; one query tile per group (d = 192, 256, and short chunks) and two (the last group has one, not whole); several
# superblocks in the last chunk (of at least 32 pairs per CTA and 32 MB: 316 entity tiles of 400 at d = 256, 512 of 1,063 at d = 128).
# Lists and ranks of a sample of the queries against the oracle.
@pytest.mark.parametrize("tiles,E,d,K", [(2, 6000, 64, 10), (2, 400_000, 128, 10), (1, 6000, 192, 3), (1, 130_000, 256, 10)])
def test_tensor_core_query_groups_share_ctas(oracle64, tiles, E, d, K):
    import kge_synth
    nq = (_shared_groups() - 1) * tiles * 128 + 70
    prob = Problem(E=E, R=9, T=100, d=d, score="distmult", B=8, N=8, P=1, graph_seed=63, tc=True)
    qh, qr, tt = kge_synth.make_queries(E, 9, nq, seed=63)
    gpu = GpuSide(prob, max_queries=nq, topk=K, load_graph=False)
    ids, sc, ranks = _infer(gpu, qh, qr, tt, K)
    some = np.unique(np.concatenate([np.arange(0, nq, 97), np.arange(127, nq, 640), [nq - 1]]))
    r_ids, r_sc, r_ranks = oracle64.score_all_topk(prob.oracle_cfg(), prob.ent, prob.rel, prob.relw, qh[some], qr[some], K + 5, true_tails=tt[some])
    for i, q in enumerate(some):
        assert len(set(ids[q])) == K
        for e in set(ids[q]) - set(r_ids[i, :K]):          # (near ties only: the sums' order differs)
            assert e in set(r_ids[i])
            f = r_sc[i][list(r_ids[i]).index(e)]
            assert abs(f - r_sc[i, K - 1]) <= 1e-4 * abs(f) + 1e-6
    assert_close(sc[some], r_sc[:, :K], atol=1e-5, what="scores")
    # (a rank moves by the entities within 2^-20 of the true tail's score: some three of 400,000)
    assert np.abs(ranks[some] - r_ranks).max() <= 2 + E // 100_000
