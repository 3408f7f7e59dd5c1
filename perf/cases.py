"""Performance cases: the decoding work that users of the library have it do.

A case is a dict of plain values.  ``prepare`` makes what a program holds
before the call (code tables, schedule, syndromes or requests, the buffers it
reuses), ``run`` is one pass through the public entry points, ``work`` counts
what the pass cannot do without.  Kinds of case:

* ``decode``: ``decode_batch`` of syndromes a program already has (a control
  loop's single shot, a handful of shots, a production batch).
* ``ler``: one chunk of a logical-error-rate curve: sample errors, make the
  greedy references, anneal (colour sweep, or the literal random-site /
  per-attempt-minimum form of the paper), decide and flag failures.
* ``batch``: a planned batch of mixed distances and noise classes.
* ``serve``: a burst of single-syndrome requests of mixed distances through
  the decode server, until every result is back.

Every output is a whole number (classes, integer energies, bit planes), so
two implementations agree exactly or not at all.
"""
import math

import numpy as np
import torch

import paper_2509_17837_gb300 as X

MIXED_DISTANCES = (5, 7, 9, 13, 17, 21)
MIXED_RESTARTS = {5: 16, 7: 16, 9: 32, 13: 32, 17: 64, 21: 64}
MIXED_SWEEPS = {5: 500, 7: 500, 9: 1000, 13: 1000, 17: 2000, 21: 2000}
SERVE_DISTANCES = (5, 9, 13, 17, 21, 25)


def _decode(name, d, shots, restarts, sweeps, p, eta, planar=False, log=False, paper_eta=False, beta0=0.05, beta1=20.0,
            scale=1024, init=1, fail=True, best_cfg=False):
    return {"name": name, "kind": "decode", "d": d, "shots": shots, "restarts": restarts, "sweeps": sweeps, "p": p,
            "eta": eta, "planar": planar, "log": log, "paper_eta": paper_eta, "beta0": beta0, "beta1": beta1,
            "scale": scale, "init": init, "fail": fail, "best_cfg": best_cfg}


def _ler(name, d, shots, p, eta, planar, literal, restarts=100, sweeps=100):
    return {"name": name, "kind": "ler", "d": d, "shots": shots, "restarts": restarts, "sweeps": sweeps, "p": p,
            "eta": eta, "planar": planar, "literal": literal}


def listed():
    return [
        # One syndrome at a time, as a control loop decodes it: the smallest
        # distance a device runs and the largest the server takes.
        _decode("one_d5", 5, 1, 32, 1000, 0.15, 100.0, fail=False),
        _decode("one_d25", 25, 1, 32, 1000, 0.15, 100.0, fail=False),
        # A handful of shots with the corrected configurations themselves.
        _decode("few_d13", 13, 16, 32, 1000, 0.15, 100.0, fail=False, best_cfg=True),
        # The small validation workload: d = 3, short anneals, many shots.
        _decode("validation_d3", 3, 1000, 8, 200, 0.10, 10.0, beta0=0.1, beta1=10.0),
        # The headline decoder settings (d = 11, 64 restarts, 1000 sweeps).
        _decode("batch_d11", 11, 4000, 64, 1000, 0.16, 100.0),
        # Larger codes in batches: depolarizing-like noise at d = 21, and the
        # strongly biased d = 31 workload at one GPU-full of chains.
        _decode("batch_d21", 21, 200, 64, 2000, 0.125, 1.0),
        _decode("batch_d31", 31, 76, 256, 2000, 0.24, 1000.0, beta0=0.02, beta1=30.0, scale=4096),
        # The paper's lattice with the paper's settings (100 restarts, 100
        # sweeps, log schedule): one chunk of a threshold curve at d = 9, the
        # same at a distance beyond the paper's, and the paper's literal
        # Metropolis form.
        _ler("curve_planar_d9", 9, 4000, 0.11, 10.0, True, False),
        _ler("curve_planar_d21", 21, 100, 0.15, 1.0, True, False),
        _ler("literal_planar_d9", 9, 500, 0.11, 10.0, True, True),
        # Mixed distances and noise classes planned as one batch.
        {"name": "mixed_batch", "kind": "batch", "shots_per_d": 250, "classes": 2},
        # A burst of requests to the decode server.
        {"name": "serve_burst", "kind": "serve", "requests": 48},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _n_stab(d, planar):
    return 2 * d * (d - 1) if planar else d * d - 1


def draw(rng):
    pick = rng.random()
    if pick < 0.06:
        return {"kind": "batch", "shots_per_d": _log_int(rng, 8, 250), "classes": rng.randint(1, 2)}
    if pick < 0.12:
        return {"kind": "serve", "requests": _log_int(rng, 1, 64)}
    d = 2 * rng.randint(1, 15) + 1
    p = round(rng.uniform(0.08, 0.20), 3)
    eta = rng.choice((1.0, 10.0, 100.0))
    if pick < 0.66:
        planar = rng.random() < 0.2
        restarts, sweeps = _log_int(rng, 4, 256), _log_int(rng, 50, 2000)
        cap = 8e9 if planar else 1e11  # attempts of one pass
        most = max(1, int(cap / (4 * restarts * sweeps * _n_stab(d, planar))))
        c = _decode(None, d, _log_int(rng, 1, min(most, 20000)), restarts, sweeps, p, eta, planar=planar,
                    init=rng.choice((0, 1, 1, 1)), fail=rng.random() < 0.5, best_cfg=rng.random() < 0.3)
    else:
        planar, literal = rng.random() < 0.6, rng.random() < 0.4
        restarts, sweeps = _log_int(rng, 8, 128), _log_int(rng, 20, 200)
        cap = 3e9 if literal else 8e9
        most = max(1, int(cap / (4 * restarts * sweeps * _n_stab(d, planar))))
        c = _ler(None, d, _log_int(rng, 1, min(most, 20000)), p, rng.choice((1.0, 5.0, 10.0)), planar, literal,
                 restarts, sweeps)
    del c["name"]
    return c


class _Held:
    """What a program keeps between calls."""


def _schedule(noise, c):
    return X.Schedule(noise, c["sweeps"], c["beta0"], c["beta1"], X.PAPER_LOG if c["log"] else X.LINEAR)


def _prepare_decode(c, seed):
    s = _Held()
    s.code = X.Code(c["d"], X.LAYOUT_PLANAR if c["planar"] else X.LAYOUT_ROTATED)
    s.noise = X.noise_from_eta(c["p"], c["eta"], X.CONVENTION_PAPER if c["paper_eta"] else X.CONVENTION_Y_OVER_XZ,
                               c["scale"])
    s.sched = _schedule(s.noise, c)
    s.seed, s.restarts, s.init, s.best_cfg = seed, c["restarts"], c["init"], c["best_cfg"]
    errors, s.syndromes = X.sample_errors(s.code, s.noise, seed, 0, c["shots"])
    s.errors = errors if c["fail"] else None
    n, dev, w = c["shots"], s.syndromes.device, 2 * s.code.words
    s.out = dict(cls=torch.empty(n, dtype=torch.uint8, device=dev),
                 E4=torch.empty((n, 4), dtype=torch.int32, device=dev),
                 recovery=torch.empty((n, w), dtype=torch.int32, device=dev),
                 best_cfg=torch.empty((n, w), dtype=torch.int32, device=dev) if s.best_cfg else None,
                 fail=torch.empty(n, dtype=torch.uint8, device=dev) if c["fail"] else None)
    s.workspace = torch.empty(X.decode_workspace_size(s.code, n, s.restarts, s.best_cfg), dtype=torch.uint8,
                              device=dev)
    return s


def _run_decode(s):
    return X.decode_batch(s.code, s.noise, s.sched, s.seed, 0, s.syndromes, s.restarts, randomised=s.init,
                          true_errors=s.errors, want_best_cfg=s.best_cfg, out=s.out, workspace=s.workspace)


def _prepare_ler(c, seed):
    s = _Held()
    s.code = X.Code(c["d"], X.LAYOUT_PLANAR if c["planar"] else X.LAYOUT_ROTATED)
    s.noise = X.noise_from_eta(c["p"], c["eta"], X.CONVENTION_PAPER, 1024)
    s.sched = X.Schedule(s.noise, c["sweeps"], 0.9, 1.0, X.PAPER_LOG)
    s.seed, s.shots, s.restarts = seed, c["shots"], c["restarts"]
    s.form = (X.ORDER_RANDOM_SITE, X.EMIN_PER_ATTEMPT) if c["literal"] else (X.ORDER_COLOUR, X.EMIN_PER_PHASE)
    return s


def _run_ler(s):
    errors, syndromes = X.sample_errors(s.code, s.noise, s.seed, 0, s.shots)
    init, cbits = X.greedy_init(s.code, s.noise, s.seed, 0, syndromes, s.restarts)
    a = X.anneal(s.code, s.sched, s.seed, 0, init, want_cfg=False, order=s.form[0], emin=s.form[1])
    r = X.decode_reduce(s.code, init, cbits, a["best_E"], true_errors=errors)
    return dict(errors=errors, syndromes=syndromes, best_E=a["best_E"], cls=r["cls"], E4=r["E4"],
                recovery=r["recovery"], fail=r["fail"])


def _prepare_batch(c, seed):
    s = _Held()
    rng = np.random.default_rng(seed)
    segments, shot0 = [], 0
    for d in MIXED_DISTANCES:
        code = X.Code(d)
        for k in range(c["classes"]):
            noise = X.noise_from_eta(0.08 + 0.005 * int(rng.integers(25)), (1.0, 10.0, 100.0)[int(rng.integers(3))])
            n = c["shots_per_d"] // c["classes"] + (k < c["shots_per_d"] % c["classes"])
            errors, syndromes = X.sample_errors(code, noise, seed, shot0, n)
            segments.append(dict(code=code, noise=noise, sched=X.Schedule(noise, MIXED_SWEEPS[d], 0.05, 20.0),
                                 shot0=shot0, syndromes=syndromes, true_errors=errors, restarts=MIXED_RESTARTS[d]))
            shot0 += n
    s.batch = X.Batch(segments, seed)
    return s


def _run_batch(s):
    s.batch.run(0)
    return s.batch.outputs


def _prepare_serve(c, seed):
    s = _Held()
    rng = np.random.default_rng(seed)
    s.server = X.Server(seed, 32, 1000, 0.05, 20.0, max_batch=1024, n_slots=8, hbm_budget_bytes=1 << 30)
    noise = X.noise_from_eta(0.15, 100.0)
    pool = []
    for d in SERVE_DISTANCES:
        cid = s.server.add_class(d, noise)
        _, syndromes = X.sample_errors(X.Code(d), noise, seed, 0, 64, want_errors=False)
        pool.append((cid, syndromes.cpu().numpy().view(np.uint32)))
    s.server.start()
    s.requests = []
    for k in range(c["requests"]):
        cid, syndromes = pool[k % len(pool)]
        s.requests.append((k, cid, np.ascontiguousarray(syndromes[int(rng.integers(64))])))
    return s


def _run_serve(s):
    n = len(s.requests)
    for req in s.requests:
        if s.server.submit(*req) != 0:
            raise RuntimeError("the server refused a request")
    got = []
    for _ in range(200):
        got += s.server.poll(cap=n, timeout_ms=100)
        if len(got) >= n:
            break
    if len(got) != n:
        raise RuntimeError("the server returned %d of %d results" % (len(got), n))
    got.sort(key=lambda r: r["req_id"])
    return dict(cls=np.array([r["cls"] for r in got], np.int64), E4=np.array([r["E4"] for r in got], np.int64),
                recovery=np.array([w for r in got for w in r["recovery"]], np.int64))


def prepare(case, seed):
    s = {"decode": _prepare_decode, "ler": _prepare_ler, "batch": _prepare_batch, "serve": _prepare_serve}[
        case["kind"]](case, seed)
    s.run = {"decode": _run_decode, "ler": _run_ler, "batch": _run_batch, "serve": _run_serve}[case["kind"]]
    return s


def run(state):
    return state.run(state)


# Integer operations of one move attempt: gather four 2-bit states, look the
# move up, compare, change the configuration and the energy, and a quarter of
# a Philox4x32-10 block.
OPS_PER_ATTEMPT = 30


def _one(d, planar, shots, restarts, sweeps):
    n_stab = _n_stab(d, planar)
    in_out = n_stab / 8 + (n_stab + 1) / 4 + 32
    return {"bytes": shots * in_out, "flops": OPS_PER_ATTEMPT * 4.0 * shots * restarts * sweeps * n_stab}


def work(case):
    if case["kind"] == "batch":
        parts = [_one(d, False, case["shots_per_d"], MIXED_RESTARTS[d], MIXED_SWEEPS[d]) for d in MIXED_DISTANCES]
    elif case["kind"] == "serve":
        parts = [_one(d, False, case["requests"] / len(SERVE_DISTANCES), 32, 1000) for d in SERVE_DISTANCES]
    else:
        parts = [_one(case["d"], case["planar"], case["shots"], case["restarts"], case["sweeps"])]
    return {k: sum(w[k] for w in parts) for k in ("bytes", "flops")}


def exact(case, seed):
    """Every output is a whole number and has to be equal; none needs a wider reference."""
    return None
