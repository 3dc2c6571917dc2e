"""Performance cases: the decodes that users of this framework run, through its public entry points.

Every case is one call on a batch of syndromes with a resident decoder: corrections, logical flips and
per-shot records, and the soft vector where it is asked for. Sizes, noise strengths and ensemble
shapes are those of the benchmark's workloads, the streaming service and the tests: code-capacity,
phenomenological and circuit-level noise on the 6.6.6 and 4.8.8 colour codes, FP32 and FP16 messages,
LSD order 0 and 5, one warp per shot or per (shot, member) pair, single problems and mixed batches,
device and host buffers.
"""
import functools
import math

import numpy as np
import torch

from paper_2508_15743_gb300 import circuit as C
from paper_2508_15743_gb300 import dem as D
from paper_2508_15743_gb300 import vibe as V

ALPHA = 0.625


def _case(name, **kw):
    """A case with the fields it does not name at their usual values."""
    c = dict(family="pheno", tiling="666", schedule="xz", noise="si1000", d="9", rounds=9, p="0.01", K=16, T=30, M=5,
             order=0, fp16=False, pair=False, flood=0, layered=0, alpha_mix=False, soft=False, entry="device", shots=1,
             sweeps=1.0)
    unknown = set(kw) - set(c)
    if unknown:
        raise KeyError(sorted(unknown))
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the plain decoder on the small code-capacity problem, with the posteriors a second stage reads:
        # a whole batch in well under a millisecond, where launches count
        _case("codecap_d5", family="codecap", d="5", p="0.05", K=1, T=20, M=1, soft=True, shots=10_000, sweeps=5.0),
        # a handful of requests of the phenomenological problem as the streaming service sends them when it is
        # not busy: latency of one small batch, members on separate warps
        _case("stream_pheno_d9", pair=True, shots=16, sweeps=260.0),
        # the headline workload: large batches of the d=9 phenomenological problem, FP32 messages
        _case("pheno_d9_f32", shots=32_768, sweeps=223.0),
        # the same with FP16 messages (FP32 marginals)
        _case("pheno_d9_f16", fp16=True, shots=32_768, sweeps=223.0),
        # the square-octagon code of the same distance, whose rows have up to 10 entries, end to end from
        # pinned host buffers
        _case("pheno488_d9_host", tiling="488", entry="host", shots=8_192, sweeps=219.0),
        # an ensemble mixing schedules (flooding, layered, serial) and scaling factors
        _case("ensemble_pheno_d7", d="7", rounds=7, p="0.012", flood=4, layered=3, alpha_mix=True, shots=6_000,
              sweeps=160.0),
        # a small circuit-level code, FP16, throughput
        _case("circuit_d5_f16", family="circuit", d="5", rounds=5, p="0.001", K=32, T=20, fp16=True, shots=4_096,
              sweeps=200.0),
        # the XYZ circuit (each ancilla cycles its measurement basis), FP32 throughput
        _case("xyz_d7_f32", family="circuit", schedule="xyz", d="7", rounds=7, p="0.001", shots=2_500, sweeps=120.0),
        # requests of the streaming service's circuit-level mix at a rate the decoder sustains: a few shots,
        # the latency of their slowest member
        _case("stream_circuit_d9_d13", family="circuit", d="9,13", rounds=0, p="0.001", K=32, T=50, fp16=True,
              pair=True, entry="mixed", shots=4, sweeps=900.0),
        # circuit-level d=11 with the large ensemble, FP32 messages
        _case("circuit_d11_f32", family="circuit", d="11", rounds=11, p="0.001", K=64, T=50, pair=True, shots=32,
              sweeps=2230.0),
        # the same with FP16 messages and the order-5 search
        _case("circuit_d11_f16_lsd5", family="circuit", d="11", rounds=11, p="0.001", K=64, T=50, order=5, fp16=True,
              pair=True, shots=32, sweeps=2230.0),
        # shots of several distances and noise strengths interleaved in one launch
        _case("mixed_circuit", family="circuit", d="5,7,9", rounds=0, p="0.001,0.003", K=32, T=20, fp16=True,
              pair=True, entry="mixed", shots=384, sweeps=420.0),
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


# Work of a pass as message updates (shots x sweeps x edges); a drawn case stays below the largest
# listed one's.
_MAX_UPDATES = 6e9


def draw(rng):
    family = rng.choice(["codecap", "pheno", "pheno", "ensemble", "circuit", "circuit", "mixed"])
    if family == "codecap":
        d = rng.choice([3, 5, 7, 9, 11, 13, 15])
        return _case("", family="codecap", tiling=rng.choice(["666", "488"]), d=str(d),
                     p=f"{_log_uniform(rng, 0.01, 0.09):.4g}", K=1, T=rng.randint(5, 30), M=1, soft=True,
                     fp16=rng.random() < 0.3, shots=int(_log_uniform(rng, 1, 20_000)), sweeps=6.0)
    if family in ("pheno", "ensemble"):
        d = rng.choice([3, 5, 7, 9])
        K = rng.randint(4, 24)
        T = rng.randint(8, 30)
        c = _case("", tiling=rng.choice(["666", "666", "488"]), d=str(d), rounds=rng.randint(2, d),
                  p=f"{_log_uniform(rng, 0.003, 0.02):.4g}", K=K, T=T, M=rng.randint(1, min(K, 7)),
                  fp16=rng.random() < 0.5, pair=rng.random() < 0.4, sweeps=0.45 * K * T,
                  order=rng.choice([0, 0, 0, 3]))
        if family == "ensemble":
            c.update(flood=rng.randint(0, K // 2), layered=rng.randint(0, K // 2), alpha_mix=rng.random() < 0.5)
        c["entry"] = rng.choice(["device", "device", "host"])
        c["shots"] = int(_log_uniform(rng, 1, 20_000))
    else:
        mixed = family == "mixed"
        K = rng.randint(4, 40)
        T = rng.randint(8, 30)
        c = _case("", family="circuit", schedule=rng.choice(["xz", "xz", "xyz"]), noise=rng.choice(["si1000", "uniform"]),
                  rounds=0, K=K, T=T, M=rng.randint(1, min(K, 7)), fp16=rng.random() < 0.6, pair=rng.random() < 0.6,
                  order=rng.choice([0, 0, 0, 5]), sweeps=0.5 * K * T)
        ds = sorted(rng.sample([3, 5, 7, 9], rng.randint(2, 3) if mixed else 1))
        ps = sorted({f"{_log_uniform(rng, 0.0007, 0.005):.4g}" for _ in range(rng.randint(1, 2) if mixed else 1)})
        c.update(d=",".join(map(str, ds)), p=",".join(ps), entry="mixed" if mixed else rng.choice(["device", "host"]))
        c["shots"] = int(_log_uniform(rng, 1, 4_000))
    # enough shots for several with a fault in them, and no more work than the largest listed case
    faults = min(1.0, min(float(dm.priors.sum()) for dm in _dems(c)))
    per_shot = c["sweeps"] * max(dm.H.nnz for dm in _dems(c))
    c["shots"] = max(math.ceil(16 / faults), min(c["shots"], int(_MAX_UPDATES / per_shot)))
    return c


@functools.lru_cache(maxsize=None)
def _dem(family, tiling, schedule, noise, d, rounds, p):
    if family == "codecap":
        return D.code_capacity_dem(d, p, tiling)
    if family == "pheno":
        return D.phenomenological_dem(d, rounds, p, p, tiling)
    return C.circuit_dem(d, rounds or d, p, noise=noise, basis="X", schedule=schedule, tiling=tiling)


def _dems(case):
    """The decoding problems of a case: one per (distance, noise strength)."""
    return [_dem(case["family"], case["tiling"], case["schedule"], case["noise"], int(d), case["rounds"], float(p))
            for d in case["d"].split(",") for p in case["p"].split(",")]


def _member_alpha(case):
    if not case["alpha_mix"]:
        return None
    mix = (0.5, 0.625, 0.75, 1.0, 0.875, 0.5625, 0.6875, 0.8125)
    return np.array([mix[i % len(mix)] for i in range(case["K"])], np.float32)


def _decoder(case, dm, i):
    perms = D.schedules(dm.n, case["K"], 100 + i, natural=case["family"] == "codecap")
    return V.Decoder(dm, case["K"], perms, T=case["T"], alpha=ALPHA, M=case["M"], lsd_order=case["order"],
                     msg_fp16=case["fp16"], n_flood=case["flood"], n_layered=case["layered"],
                     member_alpha=_member_alpha(case), pair_mode=case["pair"])


def _syndromes(case, dems, seed):
    """(problem of each shot or None, syndromes, observables) as numpy arrays."""
    B = case["shots"]
    if len(dems) == 1 and case["entry"] != "mixed":
        return (None, *D.sample(dems[0], B, seed))
    rng = np.random.default_rng(seed)
    pid = rng.permutation(np.arange(B) % len(dems)).astype(np.int32)
    syn = np.zeros((B, max(D.words(dm.m) for dm in dems)), np.uint32)
    obs = np.zeros((B, max(D.words(dm.k) for dm in dems)), np.uint32)
    for i, dm in enumerate(dems):
        rows = np.nonzero(pid == i)[0]
        if len(rows):
            s, o = D.sample(dm, len(rows), seed + 7919 * (i + 1))
            syn[rows, :s.shape[1]] = s
            obs[rows, :o.shape[1]] = o
    return pid, syn, obs


def prepare(case, seed):
    dems = _dems(case)
    pid, syn, obs = _syndromes(case, dems, seed)
    syn_t, obs_t = torch.from_numpy(syn.view(np.int32)), torch.from_numpy(obs.view(np.int32))
    decs = [_decoder(case, dm, i) for i, dm in enumerate(dems)]
    st = dict(entry=case["entry"], decoders=decs)
    B = case["shots"]
    if case["entry"] == "mixed":
        mb = V.MixedBatch(decs)
        st.update(batch=mb, problem=torch.from_numpy(pid).cuda(), syn=syn_t.cuda(), obs=obs_t.cuda(),
                  out=dict(corrections=torch.zeros((B, mb.nw), dtype=torch.int32, device="cuda"),
                           logical=torch.zeros((B, mb.kw), dtype=torch.int32, device="cuda"),
                           stats=torch.zeros((B, 12), dtype=torch.uint8, device="cuda")))
        return st
    host = case["entry"] == "host"
    dec = decs[0]

    def buffer(width, dtype):
        if host:
            return torch.zeros((B, width), dtype=dtype, pin_memory=True)
        return torch.zeros((B, width), dtype=dtype, device="cuda")

    st.update(syn=syn_t.pin_memory() if host else syn_t.cuda(), obs=obs_t.pin_memory() if host else obs_t.cuda(),
              out=dict(corrections=buffer(dec.nw, torch.int32), logical=buffer(dec.kw, torch.int32),
                       stats=buffer(12, torch.uint8),
                       soft=buffer(dec.n, torch.float32) if case["soft"] else None))
    return st


def run(state):
    out = state["out"]
    if state["entry"] == "mixed":
        return state["batch"].decode(state["problem"], state["syn"], observables=state["obs"], out=out)
    dec = state["decoders"][0]
    if state["entry"] == "host":
        V.vibe_decode_host(dec.handle, state["syn"], state["syn"].shape[0], out["corrections"], out["logical"],
                           out["stats"], state["obs"])
    else:
        dec.decode(state["syn"], observables=state["obs"], out=out)
    return {k: v for k, v in out.items() if v is not None}


def work(case):
    """Inputs and outputs once (syndromes, observables, check matrix, priors and schedules in;
    corrections, logical flips, records and soft vectors out), and for the sweeps a batch of this kind
    runs the arithmetic of every message update: the minimum, the scaling and the sums."""
    dems = _dems(case)
    by, fl = 0.0, 0.0
    for dm in dems:
        B = case["shots"] / len(dems)
        words = D.words(dm.m) + 2 * D.words(dm.k) + D.words(dm.n)
        by += B * (4 * words + 12 + (4 * dm.n if case["soft"] else 0))
        by += 4 * (dm.H.nnz + dm.m + dm.n * (1 + case["K"]))
        fl += B * case["sweeps"] * dm.H.nnz * (3 + dm.H.nnz / dm.n)
    return {"bytes": by, "flops": fl}


def exact(case, seed):
    """The soft vector of the plain decoder (one serial member in natural order) in 64 bits: the
    posteriors of the first sweep whose decision satisfies the syndrome, or after T sweeps the
    posteriors over their norm. Nothing else a case returns is a computed real number."""
    if not case["soft"] or case["K"] != 1:
        return None
    dm = _dems(case)[0]
    _, syn, _ = _syndromes(case, [dm], seed)
    s = D.unpack_bits(syn, dm.m)
    B = case["shots"]
    lam = np.log((1.0 - dm.priors) / dm.priors)
    rows = [[int(j) for j in dm.H.colidx[dm.H.rowptr[c]:dm.H.rowptr[c + 1]]] for c in range(dm.m)]
    cols = [[c for c in range(dm.m) if v in rows[c]] for v in range(dm.n)]
    H = np.zeros((dm.m, dm.n), np.uint8)
    for c in range(dm.m):
        H[c, rows[c]] = 1
    msg = {(v, c): np.full(B, lam[v]) for c in range(dm.m) for v in rows[c]}
    sign = np.where(s == 1, -1.0, 1.0)
    post = np.zeros((B, dm.n))
    soft = np.zeros((B, dm.n))
    done = np.zeros(B, bool)
    for _ in range(case["T"]):
        for v in range(dm.n):
            into = []
            for c in cols[v]:
                others = np.array([msg[u, c] for u in rows[c] if u != v]).reshape(-1, B)
                least = np.min(np.abs(others), axis=0, initial=np.inf)
                into.append(np.prod(np.where(others < 0, -1.0, 1.0), axis=0) * sign[:, c] * ALPHA * least)
            post[:, v] = lam[v] + sum(into)
            for k, c in enumerate(cols[v]):
                msg[v, c] = np.full(B, lam[v]) + sum(x for q, x in enumerate(into) if q != k)
        hit = ~done & ((((post <= 0).astype(np.uint8) @ H.T) & 1) == s).all(axis=1)
        soft[hit] = post[hit]
        done |= hit
        if done.all():
            break
    left = ~done
    soft[left] = post[left] / np.linalg.norm(post[left], axis=1, keepdims=True)
    return {"corrections": None, "logical": None, "stats": None, "soft": soft}
