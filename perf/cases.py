"""Performance cases of the library: what a user has it do, through the public binding.

Three kinds of work, each over the range it is used in:

  train     one training step (sample, gather, B x N score block, loss, backward, de-duplication, sparse row update) at the
            next step number of a run in progress: the sizes go from the 1,000-entity configuration of the tests to the batch
            of the 91-million-entity configuration.  The entity table is cut to at most two million rows: a step touches the
            2 B + N rows of its batch, and a table of a gigabyte is already far larger than the caches.
  infer     full-entity scoring: top-k tails of (h, r, ?) queries against every entity, and the rank of the true tail.
  ensemble  the power-rank fusion of many models' top-k lists.
"""
import math

import torch

import paper_2211_12281_b200 as K


def _train(name, **kw):
    case = dict(kind="train", p=1, loss="logsigmoid", opt="sgd", tc=False, gamma=12.0, temp=1.0, lr=0.05, reg=0.0, feat=0)
    case.update(kw)
    return dict(name=name, **case) if name else case


def _infer(name, **kw):
    case = dict(kind="infer", p=1, tc=False, k=10)
    case.update(kw)
    return dict(name=name, **case) if name else case


def _ensemble(name, **kw):
    case = dict(kind="ensemble", top=10, power=-0.5)
    case.update(kw)
    return dict(name=name, **case) if name else case


def listed():
    return [
        # the smallest training configuration of the repository: every launch counts
        _train("train_distmult_tiny", score="distmult", E=1000, R=10, T=20_000, d=32, B=64, N=128, P=2, gamma=0.0, temp=0.0, lr=0.1),
        # the small distance-model configuration (100,000 entities, B = N = 1,024)
        _train("train_transe_l1", score="transe", E=100_000, R=500, T=2_000_000, d=128, B=1024, N=1024, P=4),
        # sizes that are no multiple of any tile: a row width, a batch and a number of negatives picked by hand
        _train("train_rotate_ragged", score="rotate", E=100_000, R=500, T=2_000_000, d=200, B=600, N=1500, P=2),
        # shallow embeddings plus projected 768-dimensional text features, at the batch the paper quotes its step time for
        _train("train_transe_text", score="transe", E=100_000, R=500, T=2_000_000, d=256, B=512, N=1024, P=4, opt="adam", lr=0.001, feat=768),
        # sampled-softmax training on tensor cores (B = 4,096 against N = 16,384, d = 256, Adam on the touched rows)
        _train("train_complex_softmax", score="complex", E=1_000_000, R=1000, T=4_000_000, d=256, B=4096, N=16384, P=8, loss="softmax", opt="adam", lr=0.001, tc=True),
        # the large-graph batch (B = N = 8,192, d = 128, row-wise Adagrad): norm expansion on tensor cores
        _train("train_transe_l2_large", score="transe", p=2, E=2_000_000, R=1400, T=4_000_000, d=128, B=8192, N=8192, P=16, opt="adagrad", tc=True),
        # the same batch for the model whose negatives are projected per query
        _train("train_transh_l1_large", score="transh", E=2_000_000, R=1400, T=4_000_000, d=128, B=8192, N=8192, P=16, opt="adagrad"),
        # evaluation of the smallest configuration: 100 queries against 1,000 entities
        _infer("infer_distmult_tiny", score="distmult", E=1000, R=10, d=32, nq=100),
        # one serving batch: 128 queries, top-100, the row width of the paper's timing example
        _infer("infer_transe_batch", score="transe", E=1_000_000, R=1400, d=256, nq=128, k=100),
        # the validation set (15,000 queries) against a table cut to 500,000 rows, exact fp32 distances
        _infer("infer_transe_valid", score="transe", E=500_000, R=1400, d=128, nq=15_000),
        # the same queries on tensor cores against 8 M entities
        _infer("infer_distmult_valid", score="distmult", E=8_000_000, R=1400, d=128, nq=15_000, tc=True),
        # 85 models' top-100 lists for the 15,000 queries
        _ensemble("ensemble_85_models", M=85, nq=15_000, K=100),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(["train", "train_tc", "text", "infer", "infer_tc", "ensemble"], [35, 20, 10, 15, 10, 10])[0]
    if kind in ("train", "train_tc", "text"):
        if kind == "train":
            score = rng.choice(["transe", "transh", "rotate", "rotate_real_l1", "distmult", "complex"])
            p, d = rng.choice([1, 2]), 4 * rng.randint(8, 104)
        elif kind == "train_tc":
            score = rng.choice(["distmult", "complex", "transe"])
            p, d = (2 if score == "transe" else 1), 64 * rng.randint(1, 6)
        else:
            score, p, d = rng.choice(["transe", "distmult"]), rng.choice([1, 2]), 8 * rng.randint(8, 40)
        pairs_max = (1 << 26) if kind == "train_tc" else ((1 << 21) if kind == "text" else (1 << 25) * 128 // max(d, 128))
        P = rng.choice([1, 2, 4, 8])
        B = max(1, _log_int(rng, 64, 8192) // (P * P)) * P * P
        N = max(1, _log_int(rng, 128, 16384) // P) * P
        while B * N > pairs_max:
            B, N = max(1, B // 2 // (P * P)) * P * P, max(1, N // 2 // P) * P
        E = _log_int(rng, 1000, 2_000_000)
        loss, opt = rng.choice(["logsigmoid", "softmax"]), rng.choice(["sgd", "adam", "adagrad"])
        temp = rng.choice([0.0, 0.5, 1.0])
        dot = score in ("distmult", "complex")
        return _train(None, score=score, p=p, E=E, R=_log_int(rng, 10, 1400), T=min(20 * E, 4_000_000), d=d, B=B, N=N, P=P, loss=loss, opt=opt,
                      tc=kind == "train_tc", gamma=0.0 if dot else 12.0, temp=temp, lr={"sgd": min(0.05, 6.4 / B), "adam": 0.001, "adagrad": 0.05}[opt],
                      reg=rng.choice([0.0, 0.0, 1e-3]), feat=rng.choice([384, 768]) if kind == "text" else 0)
    if kind in ("infer", "infer_tc"):
        if kind == "infer":
            score = rng.choice(["transe", "transh", "rotate", "rotate_real_l1", "distmult", "complex"])
            p, d, most = rng.choice([1, 2]), 4 * rng.randint(8, 104), 15_000 * 250_000 * 128
        else:
            score, p, d, most = rng.choice(["distmult", "complex"]), 1, 64 * rng.randint(1, 6), 15_000 * 4_000_000 * 128
        nq, E = _log_int(rng, 16, 15_000), _log_int(rng, 1000, 4_000_000)
        while nq * E * d > most:
            nq, E = max(16, nq * 2 // 3), max(1000, E * 2 // 3)
        return _infer(None, score=score, p=p, E=E, R=_log_int(rng, 10, 1400), d=d, nq=nq, k=rng.choice([1, 10, 32, 100]), tc=kind == "infer_tc")
    M, k = _log_int(rng, 3, 120), rng.choice([10, 20, 50, 100])
    return _ensemble(None, M=M, nq=_log_int(rng, 100, 15_000), K=k, power=rng.choice([-1.0, -0.5, 0.5]))


# ---- inputs ----------------------------------------------------------------------------------------------------------

def _zipf(gen, n_items, s, size, dev):
    """Ranks in [0, n_items) with P(rank k) falling like (k + 1)^-s (the continuous law, rounded down)."""
    u = torch.rand(size, generator=gen, device=dev, dtype=torch.float64)
    if s == 1.0:
        x = torch.exp(u * math.log(n_items + 1.0))
    else:
        x = (1.0 - u * (1.0 - (n_items + 1.0) ** (1.0 - s))) ** (1.0 / (1.0 - s))
    return (x.long() - 1).clamp_(0, n_items - 1)


def _normal(gen, rows, width, std, dev):
    return torch.randn((rows, width), generator=gen, device=dev, dtype=torch.float32).mul_(std)


def _tables(gen, c, dev):
    """Entity rows N(0, 1/d), relation rows the same (RotatE: phases uniform in (-pi, pi)), TransH normals the same."""
    std = 1.0 / math.sqrt(c["d"])
    ent = _normal(gen, c["E"], c["d"], std, dev)
    if c["score"] in ("rotate", "rotate_real_l1"):
        rel = (torch.rand((c["R"], c["d"] // 2), generator=gen, device=dev) * 2 - 1).mul_(math.pi)
    else:
        rel = _normal(gen, c["R"], c["d"], std, dev)
    return ent, rel, _normal(gen, c["R"], c["d"], std, dev) if c["score"] == "transh" else None


def _state(gen, c, rows, width, dev):
    """Optimiser state of a run in progress: Adam's second moments of the size of a squared gradient coordinate, first
    moments below their root; row-wise Adagrad's accumulated mean squares.  A gradient coordinate is a sum of signs for
    L1 distances, of components of a unit vector for L2 ones, of table entries for the dot products."""
    if c["opt"] == "sgd":
        return None
    g = 0.03 if c["score"] in ("distmult", "complex") else (0.3 if c["p"] == 1 else 0.1)
    if c["opt"] == "adagrad":
        return torch.rand(rows, generator=gen, device=dev).add_(0.5).mul_(10 * g * g)
    s = torch.randn((rows, 2 * width), generator=gen, device=dev)
    s[:, :width].mul_(0.3 * g)
    s[:, width:].square_().add_(0.2).mul_(g * g)
    return s


def _prepare_train(c, seed, gen, dev):
    ent, rel, relw = _tables(gen, c, dev)
    kw = rel.shape[1]
    cfg = K.KgeConfig.make(num_entities=c["E"], num_relations=c["R"], dim=c["d"], score=c["score"], p_norm=c["p"], loss=c["loss"], opt=c["opt"],
                           batch=c["B"], num_neg=c["N"], num_parts=c["P"], gamma=c["gamma"], adv_temp=c["temp"],
                           ce_correction=math.log((c["E"] - 1) / c["N"]) if c["loss"] == "softmax" else 0.0, lr=c["lr"], seed=seed,
                           reg_lambda=c["reg"], prec=K.PREC_BF16_TC if c["tc"] else K.PREC_FP32, feat_dim=c["feat"])
    states = [_state(gen, c, c["E"], c["d"], dev), _state(gen, c, c["R"], kw, dev),
              _state(gen, c, c["R"], c["d"], dev) if relw is not None else None]
    kge = K.Kge(cfg)
    kge.bind(ent, rel, relw, *states, num_triples=c["T"])
    out = dict(loss=torch.zeros(1, device=dev), ent=ent, rel=rel, relw=relw, ent_state=states[0], rel_state=states[1], relw_state=states[2])
    if c["feat"]:
        std = 1.0 / math.sqrt(c["feat"])
        feat = torch.randn((c["E"], c["feat"]), generator=gen, device=dev).mul_(std).to(torch.bfloat16)
        mats = [_normal(gen, c["d"], c["feat"], 0.3 * std, dev) for _ in range(2)]
        mstates = [_state(gen, c, c["d"], c["feat"], dev) for _ in range(2)]
        kge.bind_features(feat, mats[0], mats[1], mstates[0], mstates[1])
        out.update(proj_head=mats[0], proj_tail=mats[1], proj_head_state=mstates[0], proj_tail_state=mstates[1])
    perm = torch.randperm(c["E"], generator=gen, device=dev).to(torch.int32)
    rperm = torch.randperm(c["R"], generator=gen, device=dev).to(torch.int32)
    h, t = (perm[_zipf(gen, c["E"], 1.1, c["T"], dev)] for _ in range(2))
    kge.graph_load_device(h, rperm[_zipf(gen, c["R"], 1.0, c["T"], dev)], t)
    return dict(kind="train", kge=kge, lr=c["lr"], step=1000, out=out)


def _prepare_infer(c, gen, dev):
    ent, rel, relw = _tables(gen, c, dev)
    cfg = K.KgeConfig.make(num_entities=c["E"], num_relations=c["R"], dim=c["d"], score=c["score"], p_norm=c["p"], loss="logsigmoid", opt="sgd",
                           batch=64, num_neg=64, num_parts=1, prec=K.PREC_BF16_TC if c["tc"] else K.PREC_FP32)
    kge = K.Kge(cfg)
    kge.bind(ent, rel, relw, max_queries=c["nq"], topk=c["k"])
    perm = torch.randperm(c["E"], generator=gen, device=dev).to(torch.int32)
    ids = lambda n: torch.randint(0, n, (c["nq"],), generator=gen, device=dev, dtype=torch.int32)
    return dict(kind="infer", kge=kge, k=c["k"], heads=perm[_zipf(gen, c["E"], 1.1, c["nq"], dev)], rels=ids(c["R"]), tails=ids(c["E"]),
                ids=torch.empty((c["nq"], c["k"]), dtype=torch.int32, device=dev), scores=torch.empty((c["nq"], c["k"]), device=dev),
                ranks=torch.empty(c["nq"], dtype=torch.int32, device=dev))


def _prepare_ensemble(c, gen, dev):
    # a query's models agree in part: each list is the head of one ranking of a common pool of 3 K entities plus noise of the model's own
    pool = 3 * c["K"]
    stride = 91_000_000 // pool
    ids = (torch.randint(0, stride, (c["nq"], pool), generator=gen, device=dev) + stride * torch.randperm(pool, generator=gen, device=dev)).to(torch.int32)
    common = torch.randn((c["nq"], pool), generator=gen, device=dev)
    lists = torch.empty((c["M"], c["nq"], c["K"]), dtype=torch.int32, device=dev)
    for m in range(c["M"]):
        noise = torch.randn((c["nq"], pool), generator=gen, device=dev)
        lists[m] = torch.gather(ids, 1, torch.topk(common + noise, c["K"], dim=1).indices)
    table = torch.from_numpy(K.ensemble_rank_scores(c["power"], c["K"])).to(dev)
    return dict(kind="ensemble", lists=lists, table=table, top=c["top"], ids=torch.empty((c["nq"], c["top"]), dtype=torch.int32, device=dev),
                scores=torch.empty((c["nq"], c["top"]), dtype=torch.float64, device=dev))


def prepare(case, seed):
    dev = torch.device("cuda")
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed)
    if case["kind"] == "train":
        return _prepare_train(case, seed, gen, dev)
    return _prepare_infer(case, gen, dev) if case["kind"] == "infer" else _prepare_ensemble(case, gen, dev)


# ---- one pass --------------------------------------------------------------------------------------------------------

def run(s):
    if s["kind"] == "train":        # the next step of the run: the batch of that step is drawn inside
        s["kge"].train_step(s["step"], s["lr"], loss_out=s["out"]["loss"])
        s["step"] += 1
        return s["out"]
    if s["kind"] == "infer":
        s["kge"].score_all_topk(s["heads"], s["rels"], s["k"], s["tails"], s["ids"], s["scores"], s["ranks"])
        return dict(ids=s["ids"], scores=s["scores"], ranks=s["ranks"])
    code = K.ensemble_topk(s["lists"], s["table"], s["top"], s["ids"], s["scores"])
    if code != 0:
        raise RuntimeError(f"ensemble_topk returned {code}")
    return dict(ids=s["ids"], scores=s["scores"])


# ---- what a pass cannot do without -----------------------------------------------------------------------------------

def _pair_flops(score, p):
    """Operations per (pair, coordinate) of the score: a contraction 2; |q - t| two and an addition; a complex modulus 3.5;
    TransH the projection's contraction, the residual and its norm."""
    if score in ("distmult", "complex"):
        return 2
    if score == "transh":
        return 7
    return 3.5 if score == "rotate" and p == 1 else 3


def work(case):
    c = case
    if c["kind"] == "ensemble":
        return dict(bytes=4 * c["M"] * c["nq"] * c["K"] + 12 * c["nq"] * c["top"], flops=c["M"] * c["nq"] * c["K"])
    width = c["d"]
    if c["kind"] == "infer":
        row = 2 if c["tc"] else 4
        return dict(bytes=row * c["E"] * width + c["nq"] * (12 + 8 * c["k"] + 4), flops=_pair_flops(c["score"], c["p"]) * c["nq"] * c["E"] * width)
    rows = 2 * c["B"] + c["N"]
    # a row is read and written, with its optimiser state
    per_row = {"sgd": 2 * width, "adagrad": 2 * width + 2, "adam": 6 * width}[c["opt"]]
    rel_rows = min(c["B"], c["R"]) * (2 if c["score"] == "transh" else 1)
    bytes_ = 4 * (rows + rel_rows) * per_row + 4 * (3 * c["B"] + c["N"])
    flops = 3 * _pair_flops(c["score"], c["p"]) * c["B"] * c["N"] * width
    if c["feat"]:
        matrix = {"sgd": 2 * width * c["feat"], "adagrad": 2 * width * (c["feat"] + 1), "adam": 6 * width * c["feat"]}[c["opt"]]
        bytes_ += 2 * rows * c["feat"] + 2 * 4 * matrix
        flops += 2 * 2 * rows * c["feat"] * width
    return dict(bytes=bytes_, flops=flops)


def tolerance(case):
    """Train: about four times the largest error over some fifty cases of these ranges (tables, states, projections, loss)
    against the fp64 oracle on the same inputs, whose operands are rounded where the path rounds."""
    if case["kind"] == "ensemble":
        return "exact"                      # fp64 additions of given numbers in a stated order
    if case["kind"] == "infer":
        # fp32: one accumulator per pair, coordinates ascending, as the library documents; tensor cores: fp32 sums of bf16
        # products, whose order can move a near-tie
        return {"rel": 1e-6, "max": 1e-5, "differ": 0.01} if case["tc"] else "exact"
    kinked = case["p"] == 1 and case["score"] not in ("distmult", "complex")      # a residual that rounds across zero flips a sign
    if case["feat"]:                        # bf16 features and projections: with an L1 distance their last bits flip signs
        return {"rel": 0.03, "max": 0.99} if kinked else {"rel": 2e-3, "max": 0.02}
    if case["tc"]:                          # bf16 scores' gradients
        return {"rel": 2e-4, "max": 4e-3}
    return {"rel": 5e-5, "max": 0.015} if kinked else {"rel": 4e-6, "max": 1e-4}
