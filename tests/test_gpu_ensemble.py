"""GPU parity of the power-rank ensemble (Section 3.2 "Ensemble", Eq. 2) against the oracle's brute force:
entity ids bit-exact and fp64 scores equal (both sides add the same rank scores in the same order), at the
paper's shape (85 models, top-100 lists) and fed by kge_score_all_topk at k = 100."""
import numpy as np
import pytest

import kge_synth
from parity_util import GpuSide, Problem

pytestmark = pytest.mark.gpu


def _gpu_ensemble(lists, power, top_n):
    import torch
    import paper_2211_12281_b200 as K
    dev = torch.device("cuda:0")
    M, nq, k = lists.shape
    table = torch.from_numpy(K.ensemble_rank_scores(power, k)).to(dev)
    ids = torch.full((nq, top_n), -7, dtype=torch.int32, device=dev)
    sc = torch.zeros((nq, top_n), dtype=torch.float64, device=dev)
    rc = K.ensemble_topk(torch.from_numpy(np.ascontiguousarray(lists)).to(dev), table, top_n, ids, sc)
    assert rc == 0
    torch.cuda.synchronize()
    return ids.cpu().numpy(), sc.cpu().numpy()


@pytest.mark.parametrize("M,nq,K,E", [(6, 200, 12, 60), (3, 33, 10, 4000), (85, 64, 100, 3000), (1, 5, 16, 100)])
@pytest.mark.parametrize("power", [-0.5, -1.0, 1.0, 2.0])
def test_ensemble_against_oracle(oracle64, M, nq, K, E, power):
    rng = np.random.default_rng(M * 1000 + K)
    lists = np.stack([np.stack([rng.permutation(E)[:K] for _ in range(nq)]) for _ in range(M)]).astype(np.int32)
    if M > 2:
        lists[1, :, K - 3:] = -1                        # a model that returned shorter lists
        lists[2, 0, :] = lists[0, 0, ::-1]              # mirrored ranks: exact ties decided by the id
    top_n = 10
    ids, sc = _gpu_ensemble(lists, power, top_n)
    o_ids, o_sc = oracle64.ensemble_topk(lists, power, top_n)
    assert (ids == o_ids).all()
    assert (sc == o_sc).all()


# unions up to and beyond what the first launch's table takes (768 of 1,024 slots), one, two and four passes of the larger
# table; one place per list; the longest list kept as bytes and the first that is sorted; blocks of 16 models with a remainder
@pytest.mark.parametrize("M,nq,K,E", [(33, 7, 31, 1024), (11, 150, 94, 100_000), (85, 3, 96, 1_000_000), (90, 3, 100, 1_000_000), (160, 2, 102, 1 << 30),
                                      (40, 9, 1, 12), (4, 5, 254, 300), (4, 5, 255, 300), (65, 40, 2, 5)])
@pytest.mark.parametrize("power", [-0.5, 1.0])
def test_ensemble_union_sizes(oracle64, M, nq, K, E, power):
    rng = np.random.default_rng(M + K)
    pick = (lambda: rng.permutation(E)[:K]) if E <= 300 else (lambda: rng.integers(0, E, K))
    lists = np.stack([np.stack([pick() for _ in range(nq)]) for _ in range(M)]).astype(np.int32)
    if K > 2:
        lists[0, 0, 1] = lists[0, 0, 0]                 # an entity twice in one list: both places count
        lists[:, 1, :] = -1                             # a query nobody answered
    ids, sc = _gpu_ensemble(lists, power, 10)
    o_ids, o_sc = oracle64.ensemble_topk(lists, power, 10)
    assert (ids == o_ids).all()
    assert (sc == o_sc).all()


# 20 lists of 254 places are 4,064 entries in the first block of models, several rounds of the insertion loop: an entity twice in
# one list, or a union beyond the table, is seen in the first of them by some lanes of a warp only, with rounds still to come
@pytest.mark.parametrize("twice", [True, False])
def test_ensemble_gives_up_on_a_table_with_rounds_to_come(oracle64, twice):
    rng = np.random.default_rng(7)
    M, nq, K = 20, 64, 254
    E = 260 if twice else 1_000_000
    lists = np.stack([np.stack([rng.permutation(E)[:K] if twice else rng.integers(0, E, K) for _ in range(nq)]) for _ in range(M)]).astype(np.int32)
    if twice:
        for q in range(nq):
            lists[q % 2, q, 3 + q] = lists[q % 2, q, q]
    ids, sc = _gpu_ensemble(lists, -0.5, 10)
    o_ids, o_sc = oracle64.ensemble_topk(lists, -0.5, 10)
    assert (ids == o_ids).all()
    assert (sc == o_sc).all()


@pytest.mark.parametrize("power", [-0.5, 1.0])
@pytest.mark.parametrize("union", [767, 768, 769])
def test_ensemble_union_of_exactly_what_the_table_takes(oracle64, union, power):
    rng = np.random.default_rng(union)
    M, nq, K = 85, 6, 100
    flat = np.stack([np.concatenate([rng.permutation(union) for _ in range(12)])[:M * K] for _ in range(nq)])    # 8,500 places: every id
    lists = np.ascontiguousarray(flat.reshape(nq, M, K).transpose(1, 0, 2)).astype(np.int32) + 1_000_000
    for q in range(nq):                                 # (a list across the seam of two permutations may name an id twice: make it distinct)
        for m in range(M):
            if len(set(lists[m, q])) < K:
                lists[m, q] = 1_000_000 + rng.permutation(union)[:K]
    assert all(len(np.unique(lists[:, q])) == union for q in range(nq))
    ids, sc = _gpu_ensemble(lists, power, 10)
    o_ids, o_sc = oracle64.ensemble_topk(lists, power, 10)
    assert (ids == o_ids).all() and (sc == o_sc).all()


def _ids_of_one_part(rng, n):
    """Entity ids whose multiplicative hash has the bit below the larger table's 13 slot bits clear."""
    inverse = pow(0x9E3779B1, -1, 1 << 32)
    h = np.unique(rng.integers(0, 1 << 32, 8 * n, dtype=np.uint64)) & ~np.uint64(1 << 18)
    ids = np.unique((h * np.uint64(inverse)) & np.uint64(0xffffffff))
    ids = ids[ids < (1 << 31)]
    return rng.permutation(ids)[:n].astype(np.int32)


@pytest.mark.parametrize("form", ["one pass", "two passes", "one part of two overflows", "more places than the larger table keeps"])
def test_ensemble_large_unions(oracle64, form):
    rng = np.random.default_rng(3)
    M, nq, K, top_n = (54 if form == "one pass" else 85), 4, 100, 10
    if form.startswith("one part"):
        lists = np.stack([_ids_of_one_part(rng, M * K).reshape(M, K) for _ in range(nq)], axis=1)
    else:
        lists = np.stack([rng.permutation(1 << 20)[:M * K].reshape(M, K) for _ in range(nq)], axis=1).astype(np.int32)
    if form.startswith("more"):
        top_n = 1100
    ids, sc = _gpu_ensemble(lists, -0.5, top_n)
    o_ids, o_sc = oracle64.ensemble_topk(lists, -0.5, top_n)
    assert (ids == o_ids).all() and (sc == o_sc).all()


# lists short enough for one launch (682 places), and the first that are not: an entity twice in a list, more places than
# entities, more than one warp's worth of queries
@pytest.mark.parametrize("M,K", [(2, 10), (1, 254), (22, 31), (31, 22), (33, 21)])
@pytest.mark.parametrize("power", [-1.0, 0.5])
def test_ensemble_an_entity_twice_in_short_lists(oracle64, M, K, power):
    rng = np.random.default_rng(M)
    lists = rng.integers(0, 3 * K, (M, 50, K)).astype(np.int32)
    ids, sc = _gpu_ensemble(lists, power, K + 3)
    o_ids, o_sc = oracle64.ensemble_topk(lists, power, K + 3)
    assert (ids == o_ids).all() and (sc == o_sc).all()


def test_ensemble_fewer_candidates_than_places_and_limits(oracle64):
    import torch
    import paper_2211_12281_b200 as K
    lists = np.array([[[4, 9, -1, -1]], [[9, 4, -1, -1]]], np.int32)
    ids, sc = _gpu_ensemble(lists, -0.5, 5)
    o_ids, o_sc = oracle64.ensemble_topk(lists, -0.5, 5)
    assert (ids == o_ids).all() and ids[0].tolist() == [4, 9, -1, -1, -1] and (sc == o_sc).all()
    dev = torch.device("cuda:0")
    big = torch.zeros((165, 1, 100), dtype=torch.int32, device=dev)                 # 16,500 entries per query
    table = torch.zeros(101, dtype=torch.float64, device=dev)
    out = torch.zeros((1, 10), dtype=torch.int32, device=dev)
    assert K.ensemble_topk(big, table, 10, out) == -4
    with pytest.raises(K.KgeError):
        K.ensemble_rank_scores(0.0, 10)                                              # Eq. 2 needs p != 0


def test_ensemble_of_three_scoring_functions_at_top_100(oracle32, oracle64):
    """Three models (TransE-L1, DistMult, ComplEx, their own random tables) score 40 queries against 20,000
    entities with k = 100; their lists (bit-exact against the fp32 oracle at k = 100) feed the ensemble."""
    import torch
    E, R, d, K, nq = 20000, 9, 32, 100, 40
    qh, qr, tt = kge_synth.make_queries(E, R, nq, seed=17)
    lists = []
    for m, score in enumerate(("transe", "distmult", "complex")):
        prob = Problem(E=E, R=R, T=100, d=d, score=score, p_norm=1, B=4, N=4, P=1, graph_seed=40 + m)
        gpu = GpuSide(prob, max_queries=nq, topk=K, load_graph=False)
        t, dev = gpu.torch, gpu.ent.device
        ids = t.empty((nq, K), dtype=t.int32, device=dev); sc = t.empty((nq, K), dtype=t.float32, device=dev)
        gpu.kge.score_all_topk(gpu.dev_i32(qh), gpu.dev_i32(qr), K, None, ids, sc)
        assert gpu.kge.get_status() == 0
        o_ids, _, _ = oracle32.score_all_topk(prob.oracle_cfg(), prob.ent, prob.rel, None, qh, qr, K)
        assert (ids.cpu().numpy() == o_ids).all()
        lists.append(ids.cpu().numpy())
    lists = np.stack(lists)
    ids, sc = _gpu_ensemble(lists, -0.5, 10)
    o_ids, o_sc = oracle64.ensemble_topk(lists, -0.5, 10)
    assert (ids == o_ids).all() and (sc == o_sc).all()


# one, two and four places per load (list length and the address of the lists), 64, 128 and 256 threads, eight and sixteen models
# at a time with a remainder, the last number of places that is cut by groups and the first that is not
@pytest.mark.parametrize("M,K,shift", [(25, 30, 0), (25, 31, 0), (24, 32, 0), (24, 32, 1), (24, 32, 2), (24, 33, 0), (12, 64, 0), (13, 65, 0), (13, 68, 2), (90, 12, 0), (17, 101, 0), (4, 7, 0)])
@pytest.mark.parametrize("power,top_n", [(-0.5, 16), (0.5, 17)])
def test_ensemble_places_per_load(oracle64, M, K, shift, power, top_n):
    import torch
    import paper_2211_12281_b200 as lib
    rng = np.random.default_rng(100 * M + K)
    nq, E = 33, max(3 * K, 40)
    names = rng.permutation(np.unique(rng.integers(0, 1 << 30, 2 * E)))[:E]
    lists = np.stack([np.stack([names[rng.permutation(E)[:K]] for _ in range(nq)]) for _ in range(M)]).astype(np.int32)
    lists[0, :, K - 1] = -1
    dev = torch.device("cuda:0")
    flat = torch.zeros(lists.size + shift, dtype=torch.int32, device=dev)
    view = flat[shift:].view(M, nq, K)
    view.copy_(torch.from_numpy(lists))
    table = torch.from_numpy(lib.ensemble_rank_scores(power, K)).to(dev)
    ids = torch.full((nq, top_n), -7, dtype=torch.int32, device=dev)
    sc = torch.zeros((nq, top_n), dtype=torch.float64, device=dev)
    assert lib.ensemble_topk(view, table, top_n, ids, sc) == 0
    o_ids, o_sc = oracle64.ensemble_topk(lists, power, top_n)
    assert (ids.cpu().numpy() == o_ids).all() and (sc.cpu().numpy() == o_sc).all()


# both sides of every line that the choice of kernel draws: entries per thread and threads of the single launch; list length and
# number of models of the first launch for longer lists
@pytest.mark.parametrize("M,K", [(4, 16), (5, 13), (12, 16), (13, 15), (12, 32), (11, 35), (10, 32), (9, 36), (8, 40), (4, 80), (2, 64), (2, 65), (1, 254), (2, 254),
                                 (29, 24), (28, 25), (15, 48), (14, 49), (41, 49), (40, 64), (41, 64), (41, 65), (40, 80), (41, 80), (20, 100), (21, 100), (12, 101), (13, 101),
                                 (12, 128), (13, 128), (12, 129), (4, 214), (4, 215), (3, 254)])
@pytest.mark.parametrize("power,top_n", [(-0.5, 10), (0.5, 17)])
def test_ensemble_kernel_choice(oracle64, M, K, power, top_n):
    test_ensemble_places_per_load(oracle64, M, K, 0, power, top_n)


# lists of places: the last cut by groups and the first by threads (16, 17), as many as threads and one more (64, 128, 256), more than entities
@pytest.mark.parametrize("M,K,top_n", [(6, 40, 40), (6, 40, 64), (6, 40, 65), (10, 64, 128), (10, 64, 129), (10, 100, 100), (60, 70, 128), (60, 70, 256), (60, 70, 257),
                                       (3, 254, 254), (3, 254, 900), (2, 3, 17)])
@pytest.mark.parametrize("power", [-0.5, 1.0])
def test_ensemble_long_results(oracle64, M, K, top_n, power):
    rng = np.random.default_rng(M + top_n)
    nq, E = 21, 3 * K
    lists = np.stack([np.stack([rng.permutation(E)[:K] for _ in range(nq)]) for _ in range(M)]).astype(np.int32)
    lists[:, 3] = np.arange(K)                               # the same list everywhere
    lists[:, 4] = np.roll(np.arange(K), 1)
    lists[:M // 2, 4] = np.roll(np.arange(K), 2)             # ties, decided by the id
    if M > 2:
        lists[M - 1, 5, 0] = lists[M - 1, 5, 1]              # an entity twice, behind the first block of models where there are several
    ids, sc = _gpu_ensemble(lists, power, top_n)
    o_ids, o_sc = oracle64.ensemble_topk(lists, power, top_n)
    assert (ids == o_ids).all() and (sc == o_sc).all()


# the same lists for as few queries as take large CTAs and as many as do not (four and eight per SM)
@pytest.mark.parametrize("M,K", [(6, 100), (16, 20), (13, 50), (3, 10), (85, 10), (40, 20), (25, 32), (30, 50), (40, 100), (10, 101)])
def test_ensemble_few_and_many_queries(oracle64, M, K):
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    rng = np.random.default_rng(M * K)
    some = np.stack([np.stack([rng.permutation(3 * K)[:K] for _ in range(37)]) for _ in range(M)]).astype(np.int32)
    o_ids, o_sc = oracle64.ensemble_topk(some, -0.5, 10)
    for nq in (4 * sms, 4 * sms + 1, 8 * sms, 8 * sms + 1):
        ids, sc = _gpu_ensemble(some[:, np.arange(nq) % 37], -0.5, 10)
        assert (ids == o_ids[np.arange(nq) % 37]).all() and (sc == o_sc[np.arange(nq) % 37]).all()
