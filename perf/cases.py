"""The calls this library's speed is judged by: whole propagations, served
job streams and the stateless merge / representative / overlap calls, through
the C ABI as a user's program makes them.

Three kinds of case:

* ``job``: one Algorithm 1 computation -- create a context from an observable,
  apply the circuit's layers from last to first (with the symmetry merge when
  a group is set), read <O> after every layer, count the live terms, destroy.
  With ``table`` the final operator is exported too, as a checkpoint would be.
* ``serve``: a stream of small jobs submitted to a server that stays up.
* ``canon``, ``merge``, ``sorted``: the stateless calls on device arrays of
  strings, as a program with its own term lists uses them.

Sizes follow pp_inputs (the workloads of the tests and of bench.py).
"""
import json
import math

import numpy as np
import torch

import paper_2512_12094_gb300 as pp
import pp_inputs as pi

GROUPS = {"none": pp.SYM_NONE, "zn": pp.SYM_ZN, "sn": pp.SYM_SN, "dn": pp.SYM_DN}


def listed():
    return [
        # the smallest job: all-to-all Heisenberg on 8 qubits, nothing
        # truncated, operator exported; launches and latency are what it pays
        job("heisenberg8", "heisenberg", 8, 3, "none", 0.0, -1, table=True),
        # the ring workload without merging: a table of ten thousands of
        # strings that every one of 1920 gates passes over
        job("ring32", "ring", 32, 20, "none", 1e-4, 10),
        # the same with translation merging: millions of strings
        job("ring32_zn", "ring", 32, 20, "zn", 1e-4, 10),
        # strings of two words, an odd ring, truncated by weight alone, a
        # checkpoint at the end
        job("ring101_zn", "ring", 101, 8, "zn", 0.0, 4, table=True),
        # translations of a lattice, no weight limit
        job("torus5x6", "torus", 30, 7, "torus", 1e-4, -1, lx=5),
        # 6048 gates a step over a small merged table, damped at every gate
        job("a2a64_sn_noise", "heisenberg", 64, 5, "sn", 1e-5, -1, noise=1),
        # sublayers of 630 commuting gates, merged after each
        job("xxz36_sn", "xxz", 36, 12, "sn", 0.05, -1),
        # a circuit at 256 angle sets at once, in both storage types
        job("columns64_f64", "ring", 64, 3, "none", 1e-5, -1, batch=256),
        job("columns45_f32", "ring", 45, 3, "none", 1e-5, -1, batch=100, f32=True),
        # representatives of a propagated table's strings
        dict(name="canon64_zn", kind="canon", n=64, group="zn", m=5000001, weight=10),
        # merge a term list by representatives, then its expectation value in
        # a state that is not invariant
        dict(name="merge32_zn", kind="merge", n=32, group="zn", m=1950001, weight=8),
        # two dozen requests at once on a server of eight slots
        dict(name="serve24", kind="serve", jobs=24, first=0),
    ]


def job(name, model, n, layers, group, eps, weight, lx=0, noise=0, batch=1, f32=False, table=False):
    return dict(name=name, kind="job", model=model, n=n, layers=layers, group=group, eps=eps,
                weight=weight, lx=lx, noise=noise, batch=batch, f32=f32, table=table)


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["ring", "ring", "ring", "torus", "heisenberg", "xxz", "columns", "columns",
                       "canon", "merge", "sorted", "serve"])
    if kind == "ring":
        group = rng.choice(["none", "zn", "zn", "dn"])
        if rng.random() < 0.3:  # truncated by weight alone: the number of terms follows from the circuit
            c = job("", "ring", _log_int(rng, 9, 160), _log_int(rng, 3, 6), group, 0.0,
                    rng.randint(2, 3 if group == "none" else 4), table=True)
        else:
            c = job("", "ring", _log_int(rng, 9, 160), _log_int(rng, 3, 14), group,
                    math.exp(rng.uniform(math.log(2e-4), math.log(3e-3))), rng.randint(5, 10))
    elif kind == "torus":
        lx, ly = rng.randint(3, 6), rng.randint(3, 7)
        c = job("", "torus", lx * ly, rng.randint(3, 6), "torus",
                math.exp(rng.uniform(math.log(2e-4), math.log(2e-3))), rng.choice([-1, 8]), lx=lx)
    elif kind == "heisenberg":
        noise = rng.choice([1, 1, 2])  # damping once a step keeps far more strings: fewer qubits
        c = job("", "heisenberg", _log_int(rng, 10, 64 if noise == 1 else 24), rng.randint(1, 4),
                rng.choice(["none", "sn"]) if noise == 1 else "sn",
                math.exp(rng.uniform(math.log(2e-5), math.log(1e-3))), -1, noise=noise)
    elif kind == "xxz":
        c = job("", "xxz", _log_int(rng, 8, 36), rng.randint(4, 11), "sn", rng.uniform(0.05, 0.08), -1)
    elif kind == "columns":
        c = job("", "ring", _log_int(rng, 10, 64), rng.randint(1, 2), rng.choice(["none", "zn"]), 1e-5,
                rng.choice([-1, 8]), batch=_log_int(rng, 3, 256), f32=rng.random() < 0.5)
    elif kind == "canon":
        g = rng.choice(["zn", "sn", "dn"])
        c = dict(kind="canon", n=_log_int(rng, 7, 200), group=g, m=_log_int(rng, 100000, 4000000),
                 weight=rng.choice([0, 6, 10]))
    elif kind in ("merge", "sorted"):
        n = rng.randint(9, 60)
        c = dict(kind=kind, n=n, group=rng.choice(["zn", "dn", "sn"]), m=_log_int(rng, 2000, 1500000),
                 weight=rng.randint(4, 10))
    else:
        c = dict(kind="serve", jobs=rng.randint(4, 20), first=rng.randint(1, 500))
    c.pop("name", None)
    return c


# ------------------------------------------------------------- the inputs

def _code(case):
    return pp.sym_torus(case["lx"]) if case["group"] == "torus" else GROUPS[case["group"]]


def _workload(case, seed):
    """The pp_inputs workload of a job, its angles moved by up to 1 % by the seed."""
    n, L, r = case["n"], case["layers"], np.random.default_rng(seed)
    f = 1.0 + 0.01 * r.uniform(-1.0, 1.0, 3)
    sym = _code(case)
    if case["model"] == "ring":
        wl = pi.config1_ring(n, L, 0.4 * f[0], 0.6 * f[1], 0.3 * f[2], case["eps"], case["weight"], sym)
    elif case["model"] == "torus":
        wl = pi.torus_ising(case["lx"], n // case["lx"], L, 0.4 * f[0], 0.6 * f[1], 0.3 * f[2],
                            case["eps"], case["weight"], sym)
    elif case["model"] == "xxz":
        wl = pi.xxz_all_to_all(n, 0.05 * f[0], (L + 2) // 3, eps=case["eps"], symmetry=sym, split=True)
        # the layers that are applied are the circuit's last ones
        wl.circuit.layers = wl.circuit.layers[len(wl.circuit.layers) - L:]
    elif case["noise"]:
        wl = pi.config2_all_to_all(n, 0.02 * f[0], L, 0.01, case["eps"], case["noise"], sym)
        wl.state = pi.random_product_state(n, seed)  # Neel's orbit average vanishes
    else:
        wl = pi.config0_heisenberg(n, 0.05 * f[0], L)
    return wl


def _job_inputs(case, seed):
    """(config fields, x, z, coef, [(gx, gz, theta)] in application order, bloch)."""
    wl = _workload(case, seed)
    n, B, L = case["n"], case["batch"], case["layers"]
    x, z, c = wl.observable.arrays()
    shared = {}
    layers = []
    for k in reversed(range(L)):
        sig = tuple(wl.circuit.layers[k])
        if sig not in shared:
            gx, gz, th = wl.circuit.gate_arrays(k)
            if B > 1:  # angle sets in [0, pi/2] per column, as the batched ring workload draws them
                a = pi.batched_ring_angles(B, seed)
                th = np.repeat(a.T, n, axis=0)
            shared[sig] = (gx, gz, np.ascontiguousarray(th))
        layers.append(shared[sig])
    coef = np.repeat(c[:, None], B, axis=1) if B > 1 else c
    cfg = dict(n_qubits=n, symmetry=wl.symmetry, coeff_eps=wl.eps, max_weight=wl.max_weight,
               noise_mode=wl.noise_mode, noise_p=wl.noise_p, batch=B, coef_type=int(case["f32"]))
    return cfg, x, z, coef, layers, wl.state.bloch


def _serve_workloads(case, seed):
    """Requests of the scaled serving stream: ring jobs at n = 16 to 64 (weight
    <= 8, eps >= 1e-4) and small all-to-all jobs."""
    r = np.random.default_rng(seed)
    out = []
    for j in pi.serving_stream(case["first"] + case["jobs"], seed=0)[case["first"]:]:
        a = np.array(j["angles"]) * (1.0 + 0.01 * r.uniform(-1.0, 1.0, 3))
        eps = max(j["eps"], 1e-4)
        if j["family"] == "ring":
            wl = pi.config1_ring(min(j["n"], 64), min(j["steps"], 10), a[0], a[1], a[2], eps, 8, j["group"])
        else:
            n = {16: 8, 32: 10, 64: 12, 128: 16}[j["n"]]
            wl = pi.config0_heisenberg(n, 0.02 + 0.02 * a[0], min(j["steps"], 4))
            wl.observable, wl.state = pi.mean_z(n), pi.neel_state(n)
            wl.eps, wl.symmetry = eps, j["group"]
        out.append(wl)
    return out


def _random_keys(m, n, weight, gen):
    """[m, 2W] int64 on the GPU: strings of up to `weight` letters (0: any)."""
    W, dev = (n + 63) // 64, gen.device
    k = torch.zeros(m, 2 * W, dtype=torch.int64, device=dev)
    if weight == 0:
        top = torch.iinfo(torch.int64).max
        k = torch.randint(-top, top, (m, 2 * W), generator=gen, device=dev)
        for j in range(W):
            b = n - 64 * j
            if b < 64:
                k[:, j] &= (1 << b) - 1
                k[:, W + j] &= (1 << b) - 1
        return k
    one = torch.ones(m, dtype=torch.int64, device=dev)
    for _ in range(weight):
        q = torch.randint(0, n, (m,), generator=gen, device=dev)
        p = torch.randint(1, 4, (m,), generator=gen, device=dev)
        for j in range(W):
            bit = torch.where((q >> 6) == j, one << (q & 63), 0)
            k[:, j] |= torch.where((p & 1) == 1, bit, 0)
            k[:, W + j] |= torch.where((p & 2) == 2, bit, 0)
    return k


def _term_list(case, seed):
    """A term list before a merge: random translations of m / 2 strings."""
    n, m = case["n"], case["m"]
    gen = torch.Generator("cuda").manual_seed(seed)
    base = _random_keys(max(m // 2, 1), n, case["weight"], gen)
    pick = torch.randint(0, base.shape[0], (m,), generator=gen, device="cuda")
    s = torch.randint(0, n, (m,), generator=gen, device="cuda")[:, None]
    v = base[pick]  # n <= 60: logical shifts stay inside the word
    keys = (((v << s) & ((1 << n) - 1)) | (v >> (n - s))).contiguous()
    coef = torch.randn(m, generator=gen, device="cuda", dtype=torch.float64)
    bloch = torch.from_numpy(pi.random_product_state(n, seed).bloch).cuda()
    return keys, coef, bloch


class _Server:
    """A server of eight slots that a program keeps up."""

    def __init__(self):
        self.handle = pp.pp_server_create(8, 32 << 30, 0)

    def __del__(self):
        pp.pp_server_destroy(self.handle)


def prepare(case, seed):
    if case["kind"] == "job":
        cfg, x, z, coef, layers, bloch = _job_inputs(case, seed)
        packed = {}
        for gx, gz, th in layers:
            packed.setdefault(id(th), (pp.pack_gates(gx, gz), th))
        return dict(case=case, cfg=cfg, x=x, z=z, coef=coef, bloch=bloch,
                    layers=[packed[id(l[2])] for l in layers])
    if case["kind"] == "serve":
        jobs = []
        for wl in _serve_workloads(case, seed):
            cfg = pp.pp_config_default(n_qubits=wl.circuit.n, symmetry=wl.symmetry, coeff_eps=wl.eps,
                                       max_weight=wl.max_weight)
            x, z, c = wl.observable.arrays()
            gx, gz, th = wl.circuit.gate_arrays(0)
            jobs.append(pp.make_job(cfg, x, z, c, pp.pack_gates(gx, gz), th, len(wl.circuit.layers),
                                    wl.state.bloch, True, 0))
        return dict(case=case, server=_Server(), jobs=jobs)
    if case["kind"] == "canon":
        gen = torch.Generator("cuda").manual_seed(seed)
        keys = _random_keys(case["m"], case["n"], case["weight"], gen)
        return dict(case=case, keys=keys, out=torch.empty_like(keys))
    keys, coef, bloch = _term_list(case, seed)
    return dict(case=case, keys=keys, coef=coef, bloch=bloch, keys_out=torch.zeros_like(keys),
                coef_out=torch.zeros_like(coef), out=torch.empty(1, dtype=torch.float64, device="cuda"))


# --------------------------------------------------------------- the passes

def run(s):
    case = s["case"]
    if case["kind"] == "job":
        return _run_job(s)[0]
    if case["kind"] == "serve":
        ids = [pp.pp_submit(s["server"].handle, j) for j, _ in s["jobs"]]
        res = [pp.pp_server_wait(s["server"].handle, i) for i in ids]
        bad = [r["message"] for r in res if r["status"] != 0]
        if bad:
            raise RuntimeError(bad[0])
        return {"expect": np.array([r["value"] for r in res]),
                "live": np.array([r["live_terms"] for r in res], dtype=np.int64)}
    n, m, code = case["n"], case["m"], _code(case)
    if case["kind"] == "canon":
        pp.pp_canonical_keys(n, code, m, s["keys"], s["out"])
        return s["out"]
    merge = pp.pp_merge_terms if case["kind"] == "merge" else pp.pp_merge_terms_sorted
    k = merge(n, code, m, s["keys"], s["coef"], s["keys_out"], s["coef_out"])
    if case["kind"] == "sorted":
        return {"terms": k, "keys": s["keys_out"], "coef": s["coef_out"]}  # zeros after the first k
    pp.pp_overlap_sum(n, code, k, s["keys_out"], s["coef_out"], s["bloch"], s["out"])
    return {"terms": k, "expect": s["out"]}


def _run_job(s, per_layer=None):
    case, B = s["case"], s["case"]["batch"]
    ctx = pp.pp_create(pp.pp_config_default(**s["cfg"]), s["x"], s["z"], s["coef"])
    values = []
    for gates, theta in s["layers"]:
        if per_layer is not None:
            per_layer.append(pp.pp_num_terms(ctx)[0])
        pp.pp_apply_layer(ctx, gates, theta, True)
        values.append(pp.pp_expect(ctx, s["bloch"], B))
    out = {"expect": np.array(values), "live": pp.pp_num_terms(ctx)[0]}
    if case["table"]:
        x, z, c = pp.pp_export(ctx, case["n"], B)
        # the table comes in no particular order: a checkpoint is kept sorted
        order = np.lexsort((*x.T, *z.T))
        out.update(x=x[order].view(np.int64), z=z[order].view(np.int64), coef=c[order])
    counts = None
    if per_layer is not None:
        per_layer.append(out["live"])
        counts = pp.pp_stats(ctx)
    pp.pp_destroy(ctx)
    return out, counts


_works = {}


def work(case):
    """Bytes: every layer reads the table it starts from and writes the one it
    leaves, once each (keys and coefficients of the live terms); the stateless
    calls read their arrays and write their results once.  Operations: two
    products and a sum per live anticommuting term, gate and column; one per
    letter for an overlap."""
    if case["kind"] == "canon":
        return {"bytes": 32.0 * ((case["n"] + 63) // 64) * case["m"], "flops": 0.0}
    if case["kind"] in ("merge", "sorted"):
        ov = case["n"] * case["weight"] * case["m"] / 2 if case["kind"] == "merge" else 0
        return {"bytes": 24.0 * 1.5 * case["m"], "flops": float(case["m"] + ov)}
    sig = json.dumps({k: v for k, v in case.items() if k != "name"}, sort_keys=True)
    if sig not in _works:
        total = {"bytes": 0.0, "flops": 0.0}
        if case["kind"] == "job":
            todo = [prepare(case, 0)]
        else:
            todo = [dict(case=dict(batch=1, table=False, n=wl.circuit.n), bloch=wl.state.bloch,
                         cfg=dict(n_qubits=wl.circuit.n, symmetry=wl.symmetry, coeff_eps=wl.eps,
                                  max_weight=wl.max_weight, noise_mode=0, noise_p=0.0, batch=1, coef_type=0),
                         layers=[(pp.pack_gates(gx, gz), th)] * len(wl.circuit.layers),
                         **dict(zip(("x", "z", "coef"), wl.observable.arrays())))
                    for wl in _serve_workloads(case, 0) for gx, gz, th in [wl.circuit.gate_arrays(0)]]
        for s in todo:
            live = []
            _, st = _run_job(s, live)
            row = 16 * ((s["cfg"]["n_qubits"] + 63) // 64) + (4 if s["cfg"]["coef_type"] else 8) * s["cfg"]["batch"]
            total["bytes"] += row * float(live[0] + live[-1] + 2 * sum(live[1:-1]))
            total["flops"] += 3.0 * s["cfg"]["batch"] * st["anticommuting_terms"]
        _works[sig] = total
    return dict(_works[sig])


# ------------------------------------------- the same in plain torch, 64 bits

def exact(case, seed):
    if case["kind"] == "canon":
        return None  # whole numbers
    if case["kind"] == "serve":
        return None  # thousands of layers one after the other
    if case["kind"] == "job":
        if case["batch"] > 1 and case["layers"] > 2 and case["n"] > 50:
            return None  # tens of thousands of rows of 256 columns, sorted at every gate
        return _exact_job(case, seed)
    n, code = case["n"], _code(case)
    keys, coef, bloch = _term_list(case, seed)
    dig = _canonical(_digits(keys[:, :1], keys[:, 1:], n), code)
    x, z = _words(dig)
    order = torch.argsort(x[:, 0], stable=True)
    order = order[torch.argsort(z[order, 0], stable=True)]
    both = torch.cat([z, x], 1)[order]
    first = torch.ones(len(order), dtype=torch.bool, device=both.device)
    first[1:] = (both[1:] != both[:-1]).any(1)
    run_of = torch.cumsum(first, 0) - 1
    sums = torch.zeros(int(first.sum()), dtype=torch.float64, device=both.device)
    sums.index_add_(0, run_of, coef[order])
    if case["kind"] == "sorted":
        return {"terms": None, "keys": None,
                "coef": torch.cat([sums, sums.new_zeros(case["m"] - len(sums))])}
    return {"terms": None, "expect": (sums * _overlap(dig[order][first], bloch, code)).sum().reshape(1)}


def _digits(x, z, n):
    """[m, n] letters I=0, X=1, Y=2, Z=3 of string words [m, W]."""
    q = torch.arange(n, device=x.device)
    xb, zb = (x[:, q >> 6] >> (q & 63)) & 1, (z[:, q >> 6] >> (q & 63)) & 1
    return (2 * zb + (xb ^ zb)).to(torch.uint8)


def _words(dig):
    n = dig.shape[1]
    W = (n + 63) // 64
    x = torch.zeros(dig.shape[0], W, dtype=torch.int64, device=dig.device)
    z = torch.zeros_like(x)
    for q in range(n):
        d = dig[:, q].to(torch.int64)
        x[:, q >> 6] |= ((d == 1) | (d == 2)).to(torch.int64) << (q & 63)
        z[:, q >> 6] |= (d >= 2).to(torch.int64) << (q & 63)
    return x, z


def _elements(code, n):
    """Site permutations of a group but S_n: letter q of the image is letter p[q]."""
    q = torch.arange(n)
    if code & 0xFF == pp.SYM_TORUS:
        lx = code >> 8
        return [(q % lx + dx) % lx + lx * ((q // lx + dy) % (n // lx))
                for dy in range(n // lx) for dx in range(lx)]
    rot = [(q + j) % n for j in range(n)]
    return rot + [p.flip(0) for p in rot] if code == pp.SYM_DN else rot


def _canonical(dig, code):
    """Lowest-integer member of every string's orbit, all elements tried."""
    if code == pp.SYM_NONE or dig.shape[0] == 0:
        return dig
    if code == pp.SYM_SN:
        return torch.sort(dig, dim=1, descending=True).values
    best = dig
    for p in _elements(code, dig.shape[1]):
        t = dig[:, p.to(dig.device)]
        at = dig.shape[1] - 1 - (t != best).flip(1).to(torch.uint8).argmax(1, keepdim=True)
        less = t.gather(1, at) < best.gather(1, at)
        best = torch.where(less, t, best)
    return best


def _overlap(dig, bloch, code):
    """Tr[rho s], averaged over the group's elements."""
    n = dig.shape[1]
    if code == pp.SYM_SN:
        counts = torch.stack([(dig == d).sum(1) for d in (1, 2, 3)], 1)
        kinds, back = torch.unique(counts, dim=0, return_inverse=True)
        return torch.stack([_sn_average(k.tolist(), bloch) for k in kinds])[back]
    table = torch.cat([torch.ones(n, 1, dtype=torch.float64, device=dig.device), bloch], 1)  # [n, 4]
    perms = [torch.arange(n)] if code == pp.SYM_NONE else _elements(code, n)
    out = torch.zeros(dig.shape[0], dtype=torch.float64, device=dig.device)
    for p in perms:
        t = dig[:, p.to(dig.device)].to(torch.int64)
        v = torch.ones_like(out)
        for q in range(n):
            v *= table[q][t[:, q]]
        out += v
    return out / len(perms)


def _sn_average(counts, bloch):
    """Average over all placements of counts letters: sites filled one by one."""
    n, b = bloch.shape[0], bloch.cpu().numpy()
    a = np.zeros([c + 1 for c in counts])
    a[0, 0, 0] = 1.0
    left = np.indices(a.shape)
    for k in range(n):  # a[x, y, z]: mean over placements of (x, y, z) letters on k sites
        new = a * np.maximum(k + 1 - left.sum(0), 0)
        for d in range(3):
            src = np.roll(a, 1, axis=d) * left[d] * b[k, d]
            new = new + src
        a = new / (k + 1)
    return torch.tensor(a[tuple(counts)], dtype=torch.float64, device=bloch.device)


def _parity(v):
    for s in (32, 16, 8, 4, 2, 1):
        v = v ^ (v >> s)
    return (v & 1).bool()


# i^PHASE[p, q] r is the product of letters p q
PHASE = np.zeros((4, 4), dtype=np.int64)
for _a, _b in ((1, 2), (2, 3), (3, 1)):
    PHASE[_a, _b], PHASE[_b, _a] = 1, 3


class _Table:
    """Strings (letters), a XOR-linear 63-bit hash of each, sorted by it, and
    coefficient rows.  Two strings share a hash with probability 2^-63."""

    def __init__(self, n, dev):
        r = np.random.default_rng(12345)
        self.n, self.dev = n, dev
        self.r = torch.from_numpy(r.integers(1, 2 ** 63 - 1, size=(2, n))).to(dev)  # of x bits, z bits

    def hash(self, dig):
        h = torch.zeros(dig.shape[0], dtype=torch.int64, device=self.dev)
        for q in range(self.n):
            d = dig[:, q]
            h ^= torch.where((d == 1) | (d == 2), self.r[0, q], 0)
            h ^= torch.where(d >= 2, self.r[1, q], 0)
        return h

    def put(self, dig, c, eps):
        """Equal strings added up, then truncated."""
        h, back = torch.unique(self.hash(dig), return_inverse=True)
        at = torch.zeros(len(h), dtype=torch.int64, device=self.dev)
        at[back] = torch.arange(len(back), device=self.dev)
        s = torch.zeros(len(h), c.shape[1], dtype=torch.float64, device=self.dev)
        s.index_add_(0, back, c)
        keep = (s.abs() >= eps).any(1) if eps > 0 else torch.ones(len(h), dtype=torch.bool, device=self.dev)
        self.h, self.dig, self.c = h[keep], dig[at][keep], s[keep]

    def gate(self, sites, cos, sin, eps, weight, damp):
        """sites: [(qubit, letter)]; cos, sin: [B]."""
        dig, c = self.dig, self.c
        ph = torch.ones(len(self.h), dtype=torch.int64, device=self.dev)  # i P Q
        anti = torch.zeros(len(self.h), dtype=torch.bool, device=self.dev)
        k = torch.zeros(len(self.h), dtype=torch.int64, device=self.dev)
        hp = 0
        phase = torch.from_numpy(PHASE).to(self.dev)
        for q, p in sites:
            d = dig[:, q].to(torch.int64)
            anti ^= (d != 0) & (d != p)
            ph += phase[p][d]
            k += d != 0
            hp ^= (int(self.r[0, q]) if p in (1, 2) else 0) ^ (int(self.r[1, q]) if p >= 2 else 0)
        if damp is not None:
            c = c * damp[k][:, None]
        idx = anti.nonzero()[:, 0]
        hr = self.h[idx] ^ hp
        pos = torch.searchsorted(self.h, hr).clamp(max=len(self.h) - 1)
        found = self.h[pos] == hr
        sign = torch.where((ph[idx] & 3) == 0, 1.0, -1.0).to(torch.float64)[:, None]
        other = torch.where(found[:, None], c[pos], 0.0)
        new = c.clone()
        new[idx] = cos * c[idx] - sin * sign * other
        born = idx[~found]
        child = sin * sign[~found] * c[born]
        cd = dig[born]
        flip = {0: (0, 1, 2, 3), 1: (1, 0, 3, 2), 2: (2, 3, 0, 1), 3: (3, 2, 1, 0)}
        for q, p in sites:
            cd[:, q] = torch.tensor(flip[p], dtype=torch.uint8, device=self.dev)[cd[:, q].to(torch.int64)]
        ok = torch.ones(len(born), dtype=torch.bool, device=self.dev)
        if weight >= 0:
            ok &= (cd != 0).sum(1) <= weight
        h = torch.cat([self.h, hr[~found][ok]])
        dig, new = torch.cat([dig, cd[ok]]), torch.cat([new, child[ok]])
        if eps > 0:
            keep = (new.abs() >= eps).any(1)
            h, dig, new = h[keep], dig[keep], new[keep]
        self.h, order = torch.sort(h)
        self.dig, self.c = dig[order], new[order]


def _exact_job(case, seed):
    cfg, x, z, coef, layers, bloch = _job_inputs(case, seed)
    n, code, eps, weight = case["n"], cfg["symmetry"], cfg["coeff_eps"], cfg["max_weight"]
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    as_t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev)  # noqa: E731
    t = _Table(n, dev)
    t.put(_canonical(_digits(as_t(x.view(np.int64)), as_t(z.view(np.int64)), n), code),
          as_t(np.asarray(coef, dtype=np.float64).reshape(len(coef), -1)), eps)
    p = cfg["noise_p"]
    damp = as_t((1.0 - p) ** np.arange(n + 1)) if cfg["noise_mode"] == 1 else None
    rho = as_t(np.asarray(bloch))
    # an invariant state's overlap is the same on every member of an orbit
    same = bool((rho == rho[0]).all())
    values, sites = [], {}
    for gx, gz, th in layers:
        if id(gx) not in sites:
            d = _digits(torch.from_numpy(gx.view(np.int64)), torch.from_numpy(gz.view(np.int64)), n).numpy()
            sites[id(gx)] = [[(int(q), int(r[q])) for q in np.nonzero(r)[0]] for r in d]
        cos, sin = as_t(np.cos(th).reshape(len(th), -1)), as_t(np.sin(th).reshape(len(th), -1))
        if cfg["noise_mode"] == 2:
            t.c = t.c * torch.exp(-p * (t.dig != 0).sum(1).to(torch.float64))[:, None]
            t.put(t.dig, t.c, eps)
        for g in reversed(range(len(th))):
            if len(t.h):
                t.gate(sites[id(gx)][g], cos[g], sin[g], eps, weight, damp)
        if code != pp.SYM_NONE:
            t.put(_canonical(t.dig, code), t.c, eps)
        v = (_overlap(t.dig, rho, pp.SYM_NONE if same else code)[:, None] * t.c).sum(0) if len(t.h) \
            else torch.zeros(case["batch"], dtype=torch.float64)
        values.append(v.cpu().numpy() if case["batch"] > 1 else float(v[0]))
    out = {"expect": np.array(values), "live": None}
    if case["table"]:
        xw, zw = _words(t.dig)
        xw, zw = xw.cpu().numpy().view(np.uint64), zw.cpu().numpy().view(np.uint64)
        order = np.lexsort((*xw.T, *zw.T))
        out.update(x=None, z=None, coef=t.c.cpu().numpy()[order].reshape((-1,) if case["batch"] == 1 else t.c.shape))
    return out
