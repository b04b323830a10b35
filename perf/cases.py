"""The work that users of this library have it do, as cases that can be timed.

Every case makes a seeded power-law graph (directed Chung-Lu, Zipf vertex
labels and attribute values: the family and the sizes of the workloads in
synth/) and GFDs over it, and goes through the public binding. A case is a dict:

  kind      candidates  the allocation-free candidate filter of one pattern node
            validate    one GFD: matches and sorted violations
            requests    n GFDs, one validate call each, as a serial server answers them
            batch       n GFDs in one validate_batch call, all violations fetched together
            session     n GFDs through a continuous-batching session
            load        a new graph made resident, one GFD validated on it, the graph freed
  V, E      vertices and edges; hubs: the out-degree tail of a knowledge graph
  family    star (three nodes), triangle (with a pendant chain), mixed (trees,
            cycles, 4-cliques and triangles with tails of 3 to 8 nodes), shared
            (two y of one x with two shared neighbours, and a leaf)
  n         GFDs; mode: induced, non_induced or push_x
  cap       a pattern whose expected number of matches is larger is drawn again; a
            rule without conditions (no X) reports most of its matches, so it is
            only asked for patterns a hundred times rarer
  variant   enumeration kernel kept by the program (0: the library's default)
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_2608_02321_gb300 as G

GIB = 1 << 30
MODES = {"induced": 0, "non_induced": G.FLAG_NON_INDUCED, "push_x": G.FLAG_PUSH_X}
FAMILIES = {
    # vertex labels, their Zipf exponent, edge labels, attributes, attribute values, their exponent
    "star": (8, 0.0, 4, 2, 16, 0.0),
    "triangle": (64, 1.2, 16, 4, 1024, 1.1),
    "mixed": (128, 1.2, 32, 4, 1024, 1.1),
    "shared": (500, 1.3, 64, 2, 1024, 1.1),
}


def _case(name, kind, V, E, family, n=1, mode="induced", cap=0.0, budget_gib=0, variant=0, hubs=False):
    return {"name": name, "kind": kind, "V": V, "E": E, "family": family, "n": n, "mode": mode, "cap": cap,
            "budget_gib": budget_gib, "variant": variant, "hubs": hubs}


def listed():
    return [
        # the smallest call there is: a latency-bound thread asking for one node's candidates
        _case("candidates_tiny", "candidates", 20_000, 100_000, "star"),
        # the same filter as a stream over a large vertex set
        _case("candidates_large", "candidates", 16_000_000, 32_000_000, "mixed"),
        # one selective rule on a small graph: launches and host time count
        _case("validate_star_tiny", "validate", 20_000, 100_000, "star"),
        # one cyclic rule with a chain on a mid-size graph
        _case("validate_triangle_mid", "validate", 1_000_000, 8_000_000, "triangle"),
        # requests answered one at a time with default options; one in eight is disconnected
        _case("requests_serial", "requests", 999_983, 10_000_019, "mixed", n=16, cap=1e6),
        # a rule set on a small graph: many slots, little work in each
        _case("batch_small", "batch", 10_007, 100_003, "mixed", n=64, cap=2.5e5, budget_gib=4),
        # the headline: a large rule set on a large graph, with the kernel variant that tuning picks
        _case("batch_large", "batch", 4_000_000, 40_000_000, "mixed", n=256, cap=4e7, budget_gib=48, variant=6),
        # the two semantics options, on rule sets of ordinary size
        _case("batch_push_x", "batch", 1_000_003, 10_000_000, "mixed", n=96, mode="push_x", cap=1e7, budget_gib=12),
        _case("batch_non_induced", "batch", 700_001, 5_600_000, "mixed", n=48, mode="non_induced", cap=1e6,
              budget_gib=8),
        # a knowledge-graph shape with hubs: few matches, the index build dominates
        _case("batch_kg", "batch", 5_000_000, 50_000_000, "shared", n=32, cap=1e7, budget_gib=16, hubs=True),
        # a server under load: requests admitted together, results as they finish
        _case("session", "session", 1_000_000, 10_000_000, "mixed", n=48, cap=1e6, budget_gib=16),
        # a graph that is looked at once: upload, reverse edges, one rule, free
        _case("load_validate", "load", 1_000_000, 8_000_000, "star"),
    ]


def draw(rng):
    def logu(a, b):
        return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))

    kind = rng.choice(["candidates", "validate", "requests", "batch", "batch", "session", "load"])
    if kind == "candidates":
        V = logu(10_000, 16_000_000)
        return _drawn(kind, V, 2 * V + rng.randrange(97), rng.choice(["star", "mixed"]))
    if kind == "validate":
        V = logu(10_000, 2_000_000)
        return _drawn(kind, V, V * rng.randint(5, 8) + rng.randrange(97), rng.choice(["star", "triangle"]))
    if kind == "load":
        V = logu(20_000, 1_000_000)
        return _drawn(kind, V, V * rng.randint(4, 8) + rng.randrange(97), "star")
    n = logu(8, 128) if kind == "batch" else logu(4, 32)
    V = logu(8_000, 1_000_000)
    E = V * rng.randint(7, 10) + rng.randrange(97)
    hubs = kind == "batch" and rng.random() < 0.25
    family = "shared" if hubs else "mixed"
    mode = rng.choice(["induced", "induced", "non_induced", "push_x"]) if kind == "batch" else "induced"
    cap = max(2e4, 1e6 * min(1.0, E / 1e7))
    return _drawn(kind, V, E, family, n=n, mode=mode, cap=cap, budget_gib=rng.choice([4, 8, 12]), hubs=hubs)


def _drawn(*a, **k):
    c = _case("", *a, **k)
    del c["name"]
    return c


# ---------------------------------------------------------------- inputs
def _zipf(n, values, s, gen):
    """n values in [0, values), the r-th with probability in proportion to r^-s."""
    cdf = np.cumsum(np.arange(1, values + 1, dtype=np.float64) ** -s)
    u = torch.rand(n, generator=gen, device="cuda", dtype=torch.float64) * cdf[-1]
    return torch.searchsorted(torch.from_numpy(cdf).cuda(), u, right=True).clamp_(max=values - 1).to(torch.int32)


def _power(n, count, gamma, offset, gen):
    """count vertices, the one of rank i with probability in proportion to (i + offset)^(-1/(gamma-1))."""
    b = 1.0 - 1.0 / (gamma - 1.0)
    lo, hi = offset ** b, (n + offset) ** b
    u = torch.rand(count, generator=gen, device="cuda", dtype=torch.float64)
    r = (lo + (hi - lo) * u).pow_(1.0 / b) - offset
    return r.to(torch.int64).clamp_(0, n - 1)


def _graph(case, seed):
    """The host arrays of the graph (a CSR with rows sorted by destination), and its degrees on the device."""
    V, E = case["V"], case["E"]
    n_vl, vl_s, n_el, n_at, n_av, av_s = FAMILIES[case["family"]]
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed) * 1009 + V % 997)
    place_out = torch.randperm(V, generator=gen, device="cuda")
    place_in = torch.randperm(V, generator=gen, device="cuda")
    gamma_out, off_out = (2.28, 8.0) if case["hubs"] else (2.5, 1.0)
    keys = torch.empty(0, dtype=torch.int64, device="cuda")
    while keys.numel() < E:
        more = int((E - keys.numel()) * 1.15) + 1024
        s = place_out[_power(V, more, gamma_out, off_out, gen)]
        d = place_in[_power(V, more, 2.5, 1.0, gen)]
        k = (s * V + d)[s != d]
        del s, d
        keys = torch.unique(torch.cat([keys, k]))
    if keys.numel() > E:
        keys = keys[torch.randperm(keys.numel(), generator=gen, device="cuda")[:E]].sort().values
    src = torch.div(keys, V, rounding_mode="floor")
    dst = keys - src * V
    off = torch.zeros(V + 1, dtype=torch.int64, device="cuda")
    dout = torch.bincount(src, minlength=V)
    torch.cumsum(dout, 0, out=off[1:])
    din = torch.bincount(dst, minlength=V)
    elabel = torch.randint(0, n_el, (E,), generator=gen, device="cuda", dtype=torch.int32)
    vlabel = _zipf(V, n_vl, vl_s, gen)
    attrs = torch.stack([_zipf(V, n_av, av_s, gen) for _ in range(n_at)])
    g = SimpleNamespace(n_vertices=V, out_off=off.cpu().numpy(), out_dst=dst.to(torch.int32).cpu().numpy(),
                        out_elabel=elabel.cpu().numpy(), vlabel=vlabel.cpu().numpy(), attrs=attrs.cpu().numpy())
    deg = SimpleNamespace(dout=dout.double(), din=din.double(), vlabel=vlabel, E=E, n_el=n_el, sel={}, mom={})
    return g, deg


def _moment(deg, label, a, b):
    if label not in deg.sel:
        m = slice(None) if label < 0 else deg.vlabel == label
        deg.sel[label] = (deg.dout[m], deg.din[m])
    if (label, a, b) not in deg.mom:
        o, i = deg.sel[label]
        deg.mom[label, a, b] = float((o ** a * i ** b).sum())
    return deg.mom[label, a, b]


def _expected(deg, q):
    """The expected number of maps of the pattern under the configuration model of the degrees."""
    k = len(q.node_label)
    out, inn, est = [0] * k, [0] * k, 1.0
    for s, d, l in q.edges:
        out[s] += 1
        inn[d] += 1
        est /= deg.E * (deg.n_el if l >= 0 else 1)
    for u in range(k):
        est *= _moment(deg, q.node_label[u], out[u], inn[u])
    return est


def _lit(kind, x, a, y=0, b=0, c=0):
    return SimpleNamespace(kind=kind, x=x, a=a, y=y, b=b, c=c)


def _gfd(node_label, edges, X, Y, y_false=False):
    return SimpleNamespace(node_label=node_label, edges=edges, X=X, Y=Y, y_false=y_false)


def _literal(rng, k, n_at, consts):
    x, a, y, b = (int(rng.integers(0, m)) for m in (k, n_at, k, n_at))
    return _lit(0, x, a, c=int(rng.choice(consts))) if rng.random() < 0.5 else _lit(1, x, a, y, b)


def _mixed(rng, i, label, n_el, n_at, consts):
    """A pattern of 3 to 8 nodes, 0 to 3 literals before the arrow and one behind it."""
    shape = ("tree", "cycle", "clique4", "tails")[i % 4]
    k = int(rng.integers(4 if shape == "clique4" else 3, 9))
    if shape == "cycle":
        skel = [(j, (j + 1) % k) for j in range(k)]
    else:
        core = {"tree": 1, "clique4": 4, "tails": 3}[shape]
        skel = [(a, b) for a in range(core) for b in range(a + 1, core)]
        skel += [(int(rng.integers(0, j)), j) for j in range(core, k)]
    edges = []
    for a, b in skel:
        l = -1 if rng.random() < 0.75 else int(rng.integers(0, n_el))
        edges.append((a, b, l) if rng.random() < 0.5 else (b, a, l))
    labels = [label(0.25) for _ in range(k)]
    X = [_literal(rng, k, n_at, consts) for _ in range(int(rng.integers(0, 4)))]
    return _gfd(labels, edges, X, [_literal(rng, k, n_at, consts)])


def _shared(rng, i, label, n_el, consts):
    labels = [label(0.5), label(0.0), label(0.0), label(0.5), label(0.5), -1]
    e1, e2 = (-1 if rng.random() < 0.5 else int(rng.integers(0, n_el)) for _ in range(2))
    edges = [(0, 1, e1), (0, 2, e2), (1, 3, -1), (2, 3, -1), (1, 4, -1), (2, 4, -1), (0, 5, -1)]
    if i % 2 == 0:
        return _gfd(labels, edges, [_lit(0, 1, 0, c=int(rng.choice(consts))), _lit(0, 2, 0, c=int(rng.choice(consts)))],
                    [], True)
    return _gfd(labels, edges, [], [_lit(1, 1, 0, 2, 0)])


def _disconnected(rng, g):
    """Two rare one-edge components: x -> y and z -> w, x.A0 = z.A0 implies y.A1 = w.A1."""
    freq = np.bincount(g.vlabel)
    rare = np.flatnonzero((freq > 0) & (freq <= max(8, np.sort(freq[freq > 0])[freq[freq > 0].size // 4])))
    a, b, c, d = (int(rng.choice(rare)) for _ in range(4))
    return _gfd([a, b, c, d], [(0, 1, -1), (2, 3, -1)], [_lit(1, 0, 0, 2, 0)], [_lit(1, 1, 1, 3, 1)])


def _gfds(case, seed, g, deg):
    family = case["family"]
    if family == "star":  # x(0) -[0]-> y(1), x -[1]-> z(2): y.A0 = z.A0
        return [_gfd([0, 1, 2], [(0, 1, 0), (0, 2, 1)], [], [_lit(1, 1, 0, 2, 0)])]
    if family == "triangle":  # triangle and chain on the most frequent label: x.A1 = 7 implies y.A2 = z.A2
        return [_gfd([0] * 5, [(0, 1, -1), (1, 2, -1), (0, 2, -1), (2, 3, -1), (3, 4, -1)], [_lit(0, 0, 1, c=7)],
                     [_lit(1, 1, 2, 2, 2)])]
    rng = np.random.default_rng([int(seed), 77])
    _, _, n_el, n_at, n_av, av_s = FAMILIES[family]
    freq = np.bincount(g.vlabel, minlength=8).astype(np.float64)
    top = np.argsort(-freq, kind="stable")[:8]
    p_top = freq[top] / freq[top].sum()
    p = np.arange(1, n_av + 1, dtype=np.float64) ** -av_s
    consts = rng.choice(n_av, size=4096, p=p / p.sum())

    def label(p_wild):
        return -1 if rng.random() < p_wild else int(rng.choice(top, p=p_top))

    out = []
    for i in range(case["n"]):
        if case["kind"] in ("requests", "session") and i % 8 == 7:
            out.append(_disconnected(rng, g))
            continue
        while True:
            q = _shared(rng, i, label, n_el, consts) if family == "shared" else _mixed(rng, i, label, n_el, n_at, consts)
            if _expected(deg, q) <= case["cap"] * (1.0 if q.X else 0.01):
                break
        out.append(q)
    return out


def prepare(case, seed):
    g, deg = _graph(case, seed)
    if case["kind"] == "candidates" and case["family"] == "mixed":
        gfds = [_gfd([0, -1], [(0, 1, -1)], [], [_lit(0, 0, 0, c=1)])]
    else:
        gfds = _gfds(case, seed, g, deg)
    del deg
    torch.cuda.empty_cache()
    s = SimpleNamespace(kind=case["kind"], gfds=gfds, opts={"flags": MODES[case["mode"]]})
    s.report = np.zeros(_room(case), dtype=np.int32)
    if case["budget_gib"]:
        s.opts["frontier_budget_bytes"] = case["budget_gib"] * GIB
    if case["kind"] == "load":
        s.host = g
        return s
    s.graph = G.Graph(g)
    if case["kind"] == "candidates":
        s.buf = torch.zeros(case["V"], dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
    elif case["kind"] == "batch":
        s.opts["max_violations_hint"] = 1 << 26 if case["E"] > 20_000_000 else 1 << 24
        s.opts["kernel_variant"] = case["variant"]
    elif case["kind"] == "session":
        s.session = G.Session(s.graph, max_slots=32, max_violations_hint=1 << 18, **s.opts)
    return s


# ---------------------------------------------------------------- one pass
def _room(case):
    """Ints of the report that the program keeps for violation tuples (zeros behind them, the rest left out)."""
    if case["kind"] == "candidates":
        return 0
    if case["kind"] in ("validate", "load"):
        return 1 << 20
    return 1 << 26 if case["E"] > 20_000_000 else 1 << 23


def _answers(report, results, lists=None):
    """Match and violation counts, and the sorted violations of all results back to back in the report."""
    at = 0
    for r in results if lists is None else []:
        v = r.violations().reshape(-1)[:report.size - at]
        report[at:at + v.size] = v
        at += v.size
    if lists:
        flat = lists[0].base[:report.size]  # the lists are views of one buffer, back to back
        report[:flat.size] = flat
    return {"matches": np.array([r.n_matches for r in results], dtype=np.int64),
            "violations": np.array([r.n_violations for r in results], dtype=np.int64), "tuples": report}


def run(s):
    if s.kind == "candidates":
        n = G.node_candidates_noalloc(s.graph, s.gfds[0], 0, s.buf.data_ptr(), s.buf.numel())
        return {"n": n, "ids": s.buf}
    if s.kind == "validate":
        return _answers(s.report, [s.graph.validate(s.gfds[0], **s.opts)])
    if s.kind == "requests":
        return _answers(s.report, [s.graph.validate(q) for q in s.gfds])
    if s.kind == "batch":
        results = s.graph.validate_batch(s.gfds, **s.opts)
        return _answers(s.report, results, G.violations_all(results))
    if s.kind == "session":
        ids = [s.session.submit(q) for q in s.gfds]
        got = {}
        while len(got) < len(ids):
            s.session.step()
            got.update(s.session.results())
        return _answers(s.report, [got[i] for i in ids])
    graph = G.Graph(s.host)
    return _answers(s.report, [graph.validate(s.gfds[0], **s.opts)])


def work(case):
    """Vertex data (label, both degrees) and both adjacency lists read once; for a loaded graph its host arrays."""
    V, E, n_at = case["V"], case["E"], FAMILIES[case["family"]][3]
    if case["kind"] == "candidates":
        return {"bytes": 12 * V + 4 * V // 8, "flops": 0}
    if case["kind"] == "load":
        return {"bytes": (12 + 4 * n_at) * V + 8 * E, "flops": 0}
    passes = case["n"] if case["kind"] == "requests" else 1
    return {"bytes": passes * (12 * V + 8 * E), "flops": 0}


# ---------------------------------------------------------------- the same answers, without the library
def exact(case, seed):
    """The small graphs' answers by joins over the edge list in 64-bit integers (all results are whole numbers)."""
    kind = case["kind"]
    if kind not in ("candidates", "validate") or case["E"] > 10_000_000:
        return None
    g, deg = _graph(case, seed)
    if kind == "candidates":
        need = 2 if case["family"] == "star" else 1
        v = torch.nonzero((deg.vlabel == 0) & (deg.dout >= need)).reshape(-1).to(torch.int32)
        return {"n": v.numel(), "ids": torch.nn.functional.pad(v, (0, case["V"] - v.numel()))}
    q = _gfds(case, seed, g, deg)[0]
    V = g.n_vertices
    src = np.repeat(np.arange(V, dtype=np.int64), np.diff(g.out_off))
    keys, lab = src * V + g.out_dst, g.out_elabel

    def edge(a, b):  # label of a -> b, or -2
        k = a * V + b
        at = np.minimum(np.searchsorted(keys, k), keys.size - 1)
        return np.where(keys[at] == k, lab[at], -2)

    def agrees(want, have):
        return have == -2 if want is None else (have != -2 if want < 0 else have == want)

    want = {(a, b): l for a, b, l in q.edges}
    rows = np.flatnonzero(g.vlabel == q.node_label[0]).astype(np.int64)[:, None]
    for u in range(1, len(q.node_label)):
        p = next(a for a, b, _ in q.edges if b == u)  # every later node here has an edge from an earlier one
        first, last = g.out_off[rows[:, p]], g.out_off[rows[:, p] + 1]
        cnt = last - first
        e = np.repeat(first - np.cumsum(cnt) + cnt, cnt) + np.arange(cnt.sum())
        v = g.out_dst[e].astype(np.int64)
        ok = (g.vlabel[v] == q.node_label[u]) & agrees(want[p, u], lab[e])
        rows = np.concatenate([np.repeat(rows, cnt, axis=0)[ok], v[ok, None]], axis=1)
        ok = np.ones(len(rows), dtype=bool)
        for w in range(u):
            ok &= rows[:, w] != rows[:, u]
            ok &= agrees(want.get((w, u)), edge(rows[:, w], rows[:, u]))
            ok &= agrees(want.get((u, w)), edge(rows[:, u], rows[:, w]))
        rows = rows[ok]

    def holds(l):
        a = g.attrs[l.a][rows[:, l.x]]
        return a == (l.c if l.kind == 0 else g.attrs[l.b][rows[:, l.y]])

    bad = np.ones(len(rows), dtype=bool)
    for l in q.X:
        bad &= holds(l)
    y = np.ones(len(rows), dtype=bool)
    for l in q.Y:
        y &= holds(l)
    out = rows[bad & ~y].astype(np.int32)
    flat = out[np.lexsort(out.T[::-1])].reshape(-1)
    report = np.zeros(_room(case), dtype=np.int32)
    report[:flat.size] = flat[:report.size]
    return {"matches": np.array([len(rows)], dtype=np.int64), "violations": np.array([len(out)], dtype=np.int64),
            "tuples": report}
