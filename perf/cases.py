"""What is measured: passes through the library's public calls, as verification programs make them.

A case names a network, a call and its size:

* net: the network as text, one word per ReLU layer and the logits: "1x28x28 c16k4s2p0 c32k4s2p0
  f100 f10" is a 1x28x28 input, two convolutions (channels, kernel, stride, padding) and two fully
  connected layers, a ReLU after each but the last; "3x32x32 s16 b32 b64 f100 f10" has a 3x3 stem
  and residual blocks (3x3 stride 2, 3x3, with a 1x1 stride 2 shortcut).  The networks are those of
  the synthetic workloads and tests: FC 784-100-100-10, the small and big convolution networks and
  the residual network, with He-normal weights, blurred images and margin rows y_t - y_j;
* call: deeppoly, bound, grad, opt, inter, roots or bab (see run);
* props, nodes: how many properties, and how many branch-and-bound subproblems of their rows;
* splits: ReLU splits of each subproblem; eps: radius of the input box;
* groups, group_rows: multi-neuron constraints per ReLU layer (0: none).
"""
import numpy as np
import torch
import torch.nn.functional as F

from paper_2205_00263_gb300 import Context
from paper_2205_00263_gb300.api import NodeParams

FC = "784 f100 f100 f10"
RAGGED = "2x11x11 c5k3s2p1 c7k4s2p1 f13 f4"
SMALL = "1x28x28 c16k4s2p0 c32k4s2p0 f100 f10"
BIG = "3x32x32 c32k3s1p1 c32k4s2p1 c64k3s1p1 c64k4s2p1 f512 f512 f10"
RES = "3x32x32 s16 b32 b64 f100 f10"
EPS = {FC: 0.00776, RAGGED: 0.02, SMALL: 0.00345, BIG: 0.00117, RES: 0.00234}


def _case(name, net, call, props, nodes, splits=0, steps=20, groups=0, group_rows=0, eps=None):
    return dict(name=name, net=net, call=call, props=props, nodes=nodes, splits=splits,
                steps=steps, groups=groups, group_rows=group_rows,
                eps=EPS[net] if eps is None else eps)


def listed():
    return [
        # the DeepPoly bounds of one property's rows: the smallest call, all latency
        _case("deeppoly_fc_9", FC, "deeppoly", 1, 9, splits=2),
        # bounds and minimisers' values of a few nodes of a network of odd sizes
        _case("bound_ragged_37", RAGGED, "bound", 5, 37, splits=3),
        # the subproblems of one property, as its first step or a queue that has drained has them
        _case("opt_conv_small_9", SMALL, "opt", 1, 9, splits=4),
        # the headline batch: 512 subproblems of the small convolution network, 20 Adam steps
        _case("opt_conv_small_512", SMALL, "opt", 57, 512, splits=4),
        # bound and gradient of one property's rows, the step of a caller's own optimiser
        _case("grad_conv_small_9", SMALL, "grad", 1, 9, splits=4),
        # optimised intermediate bounds at the roots of 16 properties
        _case("inter_conv_small_16", SMALL, "inter", 16, 16),
        # branch and bound of 16 fresh properties from host arrays to verdicts, 32 nodes each
        _case("bab_conv_small_16", SMALL, "bab", 16, 512),
        # the rows of one property of the FC network with multi-neuron constraints (gamma)
        _case("opt_fc_mnc_9", FC, "opt", 1, 9, splits=2, groups=16, group_rows=150),
        # a batch of the big convolution network with its constraints, about 135k rows
        _case("opt_conv_big_mnc_64", BIG, "opt", 1, 64, splits=4, groups=150, group_rows=150),
        # one bounding pass over a full batch of the big convolution network
        _case("bound_conv_big_256", BIG, "bound", 1, 256, splits=4),
        # root bounds of a new property of the big convolution network: every neuron, both sides
        _case("roots_conv_big_1", BIG, "roots", 1, 0),
        # a batch of the residual network, optimised layer by layer
        _case("opt_resnet_128", RES, "opt", 2, 128, splits=4),
    ]


def _log(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    fc = "784 " + " ".join("f%d" % _log(rng, 30, 300) for _ in range(rng.randint(1, 3))) + " f10"
    ragged = "%dx%dx%d c%dk3s2p1 c%dk4s2p1 f%d f%d" % (
        rng.randint(1, 3), rng.randint(9, 16), rng.randint(9, 16), rng.randint(3, 12),
        rng.randint(4, 16), rng.randint(10, 60), rng.randint(3, 10))
    small = "1x28x28 c%dk4s2p0 c%dk%ds2p0 f%d f10" % (
        rng.randint(6, 16), rng.randint(12, 32), rng.randint(3, 4), rng.randint(40, 120))
    big = "3x%dx%d c%dk3s1p1 c%dk4s2p1 c%dk3s1p1 c%dk4s2p1 f%d f%d f10" % (
        (rng.choice((16, 24, 32)),) * 2 + tuple(rng.choice((16, 24, 32)) for _ in range(2))
        + tuple(rng.choice((32, 48, 64)) for _ in range(2))
        + tuple(_log(rng, 100, 512) for _ in range(2)))
    res = "3x32x32 s%d b%d b%d f%d f10" % (rng.choice((8, 16)), rng.choice((16, 24, 32)),
                                           rng.choice((32, 48, 64)), rng.randint(50, 100))
    kind = rng.choice(("fc", "ragged", "small", "small", "small", "big", "big", "res"))
    net, like, most = dict(fc=(fc, FC, 512), ragged=(ragged, RAGGED, 512), small=(small, SMALL, 512),
                           big=(big, BIG, 256), res=(res, RES, 128))[kind]
    call = rng.choice(("deeppoly", "bound", "opt", "opt", "opt") + (("grad",) if kind in ("fc", "ragged", "small") else ()))
    if kind == "small":
        call = rng.choice((call, call, "inter", "bab"))
    if kind == "big":
        call = rng.choice((call, call, "roots"))
    nodes = _log(rng, 5, most)
    if call == "inter":
        nodes = _log(rng, 2, 16)
    if call == "bab":
        nodes = 32 * _log(rng, 2, 16)
    if call == "grad":
        nodes = min(nodes, 9)
    props = {"inter": nodes, "bab": nodes // 32, "roots": 1}.get(
        call, 1 if kind in ("big", "res") else max(1, min(57, nodes // 9)))
    groups = rng.randint(3, 16) if kind == "fc" and call in ("opt", "grad") and rng.random() < 0.5 else 0
    if kind == "big" and call == "opt":
        nodes = min(nodes, 64)
        groups = rng.choice((0, rng.randint(20, 150)))
    return dict(net=net, call=call, props=props, nodes=0 if call == "roots" else nodes,
                splits=0 if call in ("inter", "roots", "bab") else rng.randint(0, 6), steps=20,
                groups=groups, group_rows=rng.randint(100, 150) if groups else 0,
                eps=round(EPS[like] * rng.uniform(0.7, 1.1), 6))


# ---- the network, its properties and subproblems, from the seed alone ------------------------
def _shapes(net):
    """(input shape, affine ops): an op is (kind, source op or -1, in shape, out shape, k, s, p);
    `feeds` lists the ops that sum into each ReLU layer and into the logits."""
    words = net.split()
    shape = tuple(int(v) for v in words[0].split("x"))
    ops, feeds, src = [], [], 0  # src: ReLU layer that the next op reads (0: the input)
    shapes = [shape]

    def conv(src, co, k, s, p):
        ci, h, w = shapes[src]
        ops.append(("conv", src, (ci, h, w),
                    (co, (h + 2 * p - k) // s + 1, (w + 2 * p - k) // s + 1), k, s, p))
        return len(ops) - 1

    for w in words[1:]:
        if w[0] == "f":
            ops.append(("fc", src, shapes[src], (int(w[1:]),), 1, 1, 0))
            feed = [len(ops) - 1]
        elif w[0] == "c":
            co, rest = w[1:].split("k")
            k, rest = rest.split("s")
            s, p = rest.split("p")
            feed = [conv(src, int(co), int(k), int(s), int(p))]
        elif w[0] == "s":
            feed = [conv(src, int(w[1:]), 3, 1, 1)]
        else:  # residual block: main branch of two convolutions and a 1x1 shortcut
            first = conv(src, int(w[1:]), 3, 2, 1)
            feeds.append([first])
            shapes.append(ops[first][3])
            feed = [conv(len(feeds), int(w[1:]), 3, 1, 1), conv(src, int(w[1:]), 1, 2, 0)]
        feeds.append(feed)
        shapes.append(ops[feed[0]][3])
        src = len(feeds)
    return shape, ops, feeds


def _weights(ops, feeds, rng):
    out = []
    second = {f[0] for f in feeds if len(f) > 1}  # the second convolution of a residual branch
    for i, (kind, _, a, b, k, _, _) in enumerate(ops):
        fan = int(np.prod(a)) if kind == "fc" else a[0] * k * k
        W = rng.standard_normal((b[0], fan), dtype=np.float32) * np.float32((2.0 / fan) ** 0.5)
        if i in second:
            W *= np.float32(0.5)
        out.append((W if kind == "fc" else W.reshape(b[0], a[0], k, k),
                    (rng.standard_normal(b[0]) * 0.01).astype(np.float32)))
    return out


def _layers(ops, feeds, weights):
    """The layer list that Context.load_network takes."""
    layers, relu_at, where = [], [-1], {}
    for n, feed in enumerate(feeds):
        for o in feed:
            kind, src, a, b, k, s, p = ops[o]
            W, bias = weights[o]
            L = dict(kind=kind, W=W, b=bias, src=relu_at[src])
            if kind == "conv":
                L.update(stride=s, pad=p, in_shape=a, out_shape=b)
            layers.append(L)
            where[o] = len(layers) - 1
        if len(feed) > 1:
            layers.append(dict(kind="add", src=(where[feed[0]], where[feed[1]])))
        if n < len(feeds) - 1:
            layers.append(dict(kind="relu"))
            relu_at.append(len(layers) - 1)
    return layers


def _forward(ops, feeds, weights, x):
    """Pre-activations of every layer of images x [n, ...], in 64 bits."""
    z, pre = [x.double()], []
    for feed in feeds:
        h = 0.0
        for o in feed:
            kind, src, a, b, k, s, p = ops[o]
            W, bias = (torch.from_numpy(v).double() for v in weights[o])
            v = z[src].reshape(x.shape[0], *a)
            h = h + ((v.reshape(x.shape[0], -1) @ W.T + bias) if kind == "fc"
                     else F.conv2d(v, W, bias, s, p).reshape(x.shape[0], -1))
        pre.append(h)
        z.append(h.clamp(min=0.0))
    return pre


def _inputs(case, seed):
    """Weights, boxes, margin rows, subproblems and constraints of a case, as host arrays."""
    rng = np.random.default_rng([int(seed), 11])
    shape, ops, feeds = _shapes(case["net"])
    weights = _weights(ops, feeds, rng)
    n = case["props"]
    x = torch.from_numpy(rng.uniform(0.0, 1.0, (n,) + shape).astype(np.float32))
    if len(shape) == 3:  # 3x3 blur over the pixels within the image
        one = torch.ones(1, 1, *shape[1:])
        y = x.reshape(-1, 1, *shape[1:])
        x = (F.avg_pool2d(y, 3, 1, 1) / F.avg_pool2d(one, 3, 1, 1)).reshape(x.shape)
    pre = _forward(ops, feeds, weights, x)
    x = x.reshape(n, -1).numpy()
    eps = np.float32(case["eps"])
    lo, hi = np.maximum(0, x - eps).astype(np.float32), np.minimum(1, x + eps).astype(np.float32)
    C = []
    for p in range(n):
        y = pre[-1][p].numpy()
        t = int(np.argmax(y))
        m = np.zeros((y.size - 1, y.size), np.float32)
        for r, j in enumerate(j for j in range(y.size) if j != t):
            m[r, t], m[r, j] = 1.0, -1.0
        C.append(m)
    # constraint triples: neighbours among the neurons nearest their kink, and the rows' weights
    mnc = [[] for _ in range(n)]
    for p in range(n if case["groups"] else 0):
        for z in pre[:-1]:
            near = torch.argsort(z[p].abs()).numpy()[:min(z.shape[1], case["groups"] + 2)]
            idx = np.stack([near[:-2], near[1:-1], near[2:]], 1).repeat(case["group_rows"], 0)
            mnc[p].append((idx, rng.uniform(0.0, 1.0, idx.shape), rng.uniform(0.9, 1.1, idx.shape)))
    # subproblems: property, row, and an order in which unstable neurons are split
    R = len(feeds) - 1
    dims = [int(np.prod(ops[f[0]][3])) for f in feeds[:-1]]
    subs = []
    for i in range(case["nodes"] if case["call"] not in ("bab", "roots") else 0):
        order = rng.permutation(sum(dims))[:4000] if case["splits"] else []
        subs.append((i % n, (i // n) % C[0].shape[0], order, rng.integers(0, 2, 64) * 2 - 1))
    return dict(ops=ops, feeds=feeds, weights=weights, lo=lo, hi=hi, C=C, mnc=mnc, subs=subs, R=R,
                dims=dims)


def _facets(triples, l, u):
    """Rows over three neurons each, shaped like facets of the hull of their ReLUs:
    sum_k w_k relu(z_k) <= sum_k w_k s_k (z_k - c_k l_k), s_k the slope of neuron k's triangle and
    c_k about 1: (idx, P, Phat, p) as Context.set_mnc takes them."""
    idx, w, c = triples
    lo, hi = np.minimum(l[idx], -1e-4).astype(np.float64), np.maximum(u[idx], 1e-4).astype(np.float64)
    s = hi / (hi - lo)
    w = w / np.sqrt((w * w * (1 + s * s)).sum(1, keepdims=True))
    return (idx.astype(np.int32), w.astype(np.float32), (-w * s).astype(np.float32),
            (-w * s * c * lo).sum(1).astype(np.float32))


def _split(l, u, order, signs, count):
    """(S, l, u) of a subproblem: the first `count` neurons in `order` that are clearly unstable
    are split, sign -1 to the positive side and +1 to the negative one."""
    S, l, u = np.zeros(l.size, np.int8), l.copy(), u.copy()
    pick = [j for j in order if l[j] < -1e-3 and u[j] > 1e-3][:count]
    for j, s in zip(pick, signs):
        S[j] = s
        if s < 0:
            l[j] = 0.0
        else:
            u[j] = 0.0
    return S, l, u


def prepare(case, seed):
    """A context with the network loaded, and what the call works on: the properties' boxes and
    rows, and for calls on subproblems the nodes with their splits and constraints."""
    inp = _inputs(case, seed)
    call, SD = case["call"], sum(inp["dims"])
    E = sum(len(v[0]) for v in inp["mnc"][0])
    cap = {"roots": 2048, "bab": 8192, "inter": 1024}.get(call, max(64, 2 * case["nodes"] + 12 * case["props"]))
    ctx = Context(device=0, node_capacity=cap, max_mnc_rows=E)
    net = ctx.load_network(_layers(inp["ops"], inp["feeds"], inp["weights"]))
    s = dict(case=case, ctx=ctx, net=net, SD=SD, E=E, lo=inp["lo"], hi=inp["hi"], C=inp["C"])
    if call in ("bab", "roots"):
        return s
    s["props"] = [ctx.set_property(net, inp["lo"][p], inp["hi"][p], inp["C"][p])
                  for p in range(case["props"])]
    for p, layers in zip(s["props"], inp["mnc"]):
        for t, rows in enumerate(layers):
            ctx.set_mnc(p, t + 1, *_facets(rows, *ctx.root_bounds(p, t + 1)))
    s["rows"] = [(s["props"][p], r) for p, r, _, _ in inp["subs"]]
    if call == "inter":
        return s
    s["nodes"] = []
    for (p, r), (_, _, order, signs) in zip(s["rows"], inp["subs"]):
        node = ctx.node_root(p, r)
        if case["splits"]:
            q = ctx.export_params(node)
            S, l, u = _split(q.l, q.u, order, signs, case["splits"])
            ctx.import_params(node, NodeParams(inp["R"], inp["R"], l, u, S, q.alpha, q.beta, q.gamma))
        s["nodes"].append(node)
    return s


def run(s):
    case, ctx = s["case"], s["ctx"]
    call = case["call"]
    if call == "deeppoly":
        return ctx.deeppoly_batch(s["nodes"])
    if call == "bound":
        return ctx.bound_batch(s["nodes"])
    if call == "grad":
        return ctx.bound_grad(s["nodes"], s["SD"], s["E"])
    if call == "opt":
        # the best bound of the iterates, and the bound at the parameters the nodes now hold
        best = ctx.optimize(s["nodes"], steps=case["steps"], eps_rel=1e-3 if s["E"] else 0.0)
        return best, ctx.bound_batch(s["nodes"], with_ub=False)
    if call == "inter":
        nodes = [ctx.node_root(p, r) for p, r in s["rows"]]
        ctx.optimize_intermediate(nodes, steps=case["steps"])
        out = [ctx.export_params(n) for n in nodes]
        for n in nodes:
            ctx.node_free(n)
        return {"l": np.stack([q.l for q in out]), "u": np.stack([q.u for q in out])}
    props = [ctx.set_property(s["net"], s["lo"][p], s["hi"][p], s["C"][p])
             for p in range(case["props"])]
    if call == "roots":
        return [ctx.root_bounds(props[0], t + 1) for t in range(s["net"].R)]
    for p in props:
        ctx.set_budget(p, 32)
    while ctx.bab_step(props, max_nodes=512, steps=case["steps"])["nodes_bounded"]:
        pass
    done = [ctx.verdict(p)[:2] for p in props]
    return {"verdict": np.array([v for v, _ in done]), "bound": np.array([b for _, b in done], np.float32)}


def work(case):
    shape, ops, feeds = _shapes(case["net"])
    dims = [int(np.prod(ops[f[0]][3])) for f in feeds]
    d0, SD, R = int(np.prod(shape)), sum(dims[:-1]), len(feeds) - 1
    macs = [sum(int(np.prod(ops[o][3])) * (int(np.prod(ops[o][2])) if ops[o][0] == "fc"
                                           else ops[o][2][0] * ops[o][4] ** 2) for o in f)
            for f in feeds]  # of one row through the edges into each layer
    weights = 4.0 * sum(ops[o][3][0] * (int(np.prod(ops[o][2])) if ops[o][0] == "fc"
                                        else ops[o][2][0] * ops[o][4] ** 2) for f in feeds for o in f)
    E = min(SD, case["groups"]) and sum(min(d - 2, case["groups"]) for d in dims[:-1]) * case["group_rows"]
    sweep = 2.0 * (sum(macs[:R]) + dims[R - 1] + d0)
    n, call, boxes = case["nodes"], case["call"], 8.0 * d0 * case["props"]
    state = n * (17.0 * SD + 4.0 * E) + case["props"] * 28.0 * E  # l, u, alpha, beta, S, gamma; rows
    if call == "deeppoly":
        return dict(flops=n * sweep, bytes=weights + boxes + n * 9.0 * SD)
    if call == "bound":
        return dict(flops=2 * n * sweep, bytes=weights + boxes + state)
    if call == "grad":
        return dict(flops=n * (2 * sweep + 12.0 * E), bytes=weights + boxes + state + n * (8.0 * SD + 4.0 * E))
    if call == "opt":
        k = case["steps"]
        return dict(flops=n * ((2 * k + 3) * sweep + (k + 1) * 24.0 * E),
                    bytes=weights + boxes + state + n * (8.0 * SD + 4.0 * E))
    # rows of each layer carried to the input: a convolution neuron reaches its window only
    win = [2.0 * macs[0] / dims[0]]
    for t in range(1, R):
        h = 0.0
        if ops[feeds[t][0]][0] == "fc":
            h = 2.0 * (dims[t - 1] + sum(macs[:t]))
        else:
            side = ops[feeds[t][0]][4]
            h = 2.0 * ops[feeds[t][0]][2][0] * side * side
            for q in range(t - 1, -1, -1):
                o = ops[feeds[q][0]]
                h += 2.0 * min(side, o[3][1]) * min(side, o[3][2]) * o[3][0] * o[2][0] * o[4] ** 2
                side = (side - 1) * o[5] + o[4]
        win.append(h)
    roots = sum(2.0 * d * w for d, w in zip(dims, win))
    if call == "roots":
        return dict(flops=roots, bytes=weights + boxes + 8.0 * SD)
    if call == "inter":  # a tenth of the neurons unstable, 21 sweeps and 20 adjoints of each side
        rows = sum(0.2 * d * w for d, w in zip(dims[1:R], win[1:]))
        return dict(flops=n * (2 * case["steps"] + 1) * rows, bytes=weights + boxes + n * 16.0 * SD)
    # bab: roots, then 21 sweeps and 20 adjoints of each bounded node
    return dict(flops=case["props"] * roots + n * (2 * case["steps"] + 1) * sweep,
                bytes=weights + boxes + n * 25.0 * SD)


# ---- the same results in 64 bits -------------------------------------------------------------
class _Net64:
    def __init__(self, inp, dev):
        self.ops, self.feeds, self.R, self.dims = inp["ops"], inp["feeds"], inp["R"], inp["dims"]
        self.W = [(torch.from_numpy(w).to(dev).double(), torch.from_numpy(b).to(dev).double())
                  for w, b in inp["weights"]]
        self.off = np.concatenate([[0], np.cumsum(self.dims)]).tolist()

    def back(self, o, a):
        """Coefficients a on the op's outputs -> (coefficients on its inputs, a . bias)."""
        kind, _, i, b, k, s, p = self.ops[o]
        W, bias = self.W[o]
        if kind == "fc":
            return a @ W, a @ bias
        v = a.reshape(a.shape[0], b[0], -1)
        cols = W.reshape(b[0], -1).T @ v
        return (F.fold(cols, i[1:], k, padding=p, stride=s).reshape(a.shape[0], -1),
                v.sum(2) @ bias)

    def layer(self, v, t):
        return v[:, self.off[t - 1]:self.off[t]]

    def sweep(self, t, ahat, lo, hi, l, u, alpha, S=None, beta=None, G=None, Gh=None):
        """Lower bounds of rows of coefficients ahat on zhat_t (or, t = R + 1, on z_R)."""
        c, lam = 0.0, {}
        if t == self.R + 1:
            lam[self.R], todo = ahat, self.R
        else:
            lam[t], todo = ahat, t
        for v in range(todo, 0, -1):
            if v not in lam:
                continue
            a = lam.pop(v)
            if v < t:
                lv, uv = self.layer(l, v), self.layer(u, v)
                if G is not None:
                    a = a + self.layer(G, v)
                up = uv / torch.where(uv - lv > 0, uv - lv, torch.ones_like(uv))
                on = lv >= 0
                off = (uv <= 0) & ~on
                if S is not None:
                    sv = self.layer(S, v)
                    on = (on & (sv != 1)) | (sv == -1)
                    off = (off & (sv != -1)) | (sv == 1)
                D = torch.where(a >= 0, self.layer(alpha, v), up)
                D = torch.where(on, torch.ones_like(D), torch.where(off, torch.zeros_like(D), D))
                c = c + torch.where(~on & ~off & (a < 0), -a * up * lv, torch.zeros_like(a)).sum(1)
                a = a * D
                if beta is not None:
                    a = a + self.layer(beta, v) * sv
                if Gh is not None:
                    a = a + self.layer(Gh, v)
            for o in self.feeds[v - 1]:
                src = self.ops[o][1]
                b, off_c = self.back(o, a)
                c = c + off_c
                lam[src] = lam[src] + b if src in lam else b
        a = lam[0]
        x = torch.where(a >= 0, lo, hi)
        return c + (a * x).sum(1), x.detach()

    def value(self, x):
        z = [x]
        for feed in self.feeds[:-1]:
            h = 0.0
            for o in feed:
                kind, src, i, b, k, s, p = self.ops[o]
                W, bias = self.W[o]
                if kind == "fc":
                    h = h + z[src] @ W.T + bias
                else:
                    cols = F.unfold(z[src].reshape(-1, *i), k, padding=p, stride=s)
                    h = h + (W.reshape(b[0], -1) @ cols + bias[:, None]).reshape(x.shape[0], -1)
            z.append(h.clamp(min=0.0))
        return z[-1]

    def roots(self, lo, hi):
        """DeepPoly bounds (l, u) [SD] of every ReLU layer over one box."""
        SD = self.off[-1]
        l = torch.zeros(1, SD, dtype=torch.float64, device=lo.device)
        u, al = torch.zeros_like(l), torch.zeros_like(l)
        for t in range(1, self.R + 1):
            d, o = self.dims[t - 1], self.off[t - 1]
            per = max(1, min(d, (1 << 25) // max(self.dims)))
            for j in range(0, d, per):
                eye = torch.zeros(min(per, d - j), d, dtype=torch.float64, device=lo.device)
                eye[torch.arange(eye.shape[0]), j + torch.arange(eye.shape[0])] = 1.0
                at = slice(o + j, o + j + eye.shape[0])
                l[0, at] = self.sweep(t, eye, lo, hi, l, u, al)[0]
                u[0, at] = -self.sweep(t, -eye, lo, hi, l, u, al)[0]
            al[0, o:o + d] = (u[0, o:o + d] >= -l[0, o:o + d]).double()
        return l[0], u[0]


def _adam(params, grads, state, k, lr, eps, eps_rel):
    """One step of projected Adam, ascending; alpha to [0, 1], the others to >= 0."""
    with torch.no_grad():
        if eps_rel:
            top = torch.stack([g.abs().amax(1) for g in grads if g.shape[1]]).amax(0)
            eps = torch.clamp(eps_rel * top, min=eps)[:, None]
        for i, (p, g) in enumerate(zip(params, grads)):
            m, v = state[i]
            m.mul_(0.9).add_(g, alpha=0.1)
            v.mul_(0.999).addcmul_(g, g, value=0.001)
            p += lr[i] * (m / (1 - 0.9 ** k)) / ((v / (1 - 0.999 ** k)).sqrt() + eps)
            p.clamp_(0.0, 1.0 if i == 0 else None)


def exact(case, seed):
    if case["call"] == "bab":  # a tree: its verdicts are whole numbers
        return None
    with torch.enable_grad():
        return _exact(case, seed)


def _exact(case, seed):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    inp = _inputs(case, seed)
    net = _Net64(inp, dev)
    up = lambda v: torch.from_numpy(np.ascontiguousarray(v)).to(dev).double()  # noqa: E731
    lo, hi = up(inp["lo"]), up(inp["hi"])
    roots = [net.roots(lo[p], hi[p]) for p in range(case["props"])]
    call, off, R = case["call"], net.off, net.R
    if call == "roots":
        l, u = (v.cpu().numpy() for v in roots[0])
        return [(l[off[t]:off[t + 1]], u[off[t]:off[t + 1]]) for t in range(R)]
    of = [p for p, _, _, _ in inp["subs"]]
    lo, hi = lo[of], hi[of]
    if call == "inter":
        return _inter(net, case, lo, hi, torch.stack([roots[p][0] for p in of]),
                      torch.stack([roots[p][1] for p in of]))
    host = [tuple(v.cpu().numpy() for v in r) for r in roots]
    nodes = [_split(*host[p], order, signs, case["splits"]) if case["splits"]
             else (np.zeros(off[-1], np.int8),) + host[p] for p, _, order, signs in inp["subs"]]
    S, l, u = (up(np.stack([n[k] for n in nodes])) for k in range(3))
    l0, u0 = torch.stack([roots[p][0] for p in of]), torch.stack([roots[p][1] for p in of])
    alpha = (u0 >= -l0).double()
    WL, bL = net.W[net.feeds[-1][0]]
    C = up(np.stack([inp["C"][p][r] for p, r, _, _ in inp["subs"]]))
    A, b = C @ WL, C @ bL
    if call == "deeppoly":
        alpha = (u >= -l).double()
        return (net.sweep(R + 1, A, lo, hi, l, u, alpha, S)[0] + b).cpu().numpy()
    beta = torch.zeros_like(alpha)
    n, E = len(nodes), sum(len(v[0]) for v in inp["mnc"][0])
    gamma = torch.zeros(n, E, dtype=torch.float64, device=dev)
    maps = []  # per property: gamma -> (gamma^T P, gamma^T Phat) as sparse [SD, E], and p
    for p in range(case["props"] if E else 0):
        rows = [_facets(v, *(w[off[t]:off[t + 1]] for w in host[p])) for t, v in enumerate(inp["mnc"][p])]
        r = np.concatenate([off[t] + v[0].reshape(-1) for t, v in enumerate(rows)])
        where = torch.from_numpy(np.stack([r, np.arange(E).repeat(3)]).astype(np.int64)).to(dev)
        maps.append([torch.sparse_coo_tensor(where, up(np.concatenate([v[k].reshape(-1) for v in rows])),
                                             (off[-1], E)).coalesce() for k in (1, 2)]
                    + [up(np.concatenate([v[3] for v in rows]))])
    pick = [torch.tensor([i for i, q in enumerate(of) if q == p], device=dev) for p in range(len(maps))]

    def bound(alpha, beta, gamma):
        G = Gh = None
        cost = 0.0
        if E:
            G, Gh, cost = torch.zeros_like(alpha), torch.zeros_like(alpha), torch.zeros_like(alpha[:, 0])
            for (P, Ph, off_p), rows in zip(maps, pick):
                G = G.index_copy(0, rows, torch.sparse.mm(P, gamma[rows].T).T)
                Gh = Gh.index_copy(0, rows, torch.sparse.mm(Ph, gamma[rows].T).T)
                cost = cost.index_copy(0, rows, gamma[rows] @ off_p)
        v, x = net.sweep(R + 1, A, lo, hi, l, u, alpha, S, beta, G, Gh)
        return v + b - cost, x

    params = [alpha, beta, gamma]

    def step():
        ps = [v.detach().requires_grad_(True) for v in params]
        lb, x = bound(*ps)
        g = torch.autograd.grad(lb.sum(), ps, allow_unused=True)
        return lb.detach(), x, [torch.zeros_like(v) if w is None else w for v, w in zip(ps, g)]

    def last():
        with torch.no_grad():
            lb, x = bound(*params)
            return lb.cpu().numpy(), ((net.value(x) * A).sum(1) + b).cpu().numpy()

    if call == "bound":
        return last()
    if call == "grad":
        lb, _, g = step()
        return (lb.cpu().numpy(),) + tuple(v.cpu().numpy() for v in g)
    best = torch.full((n,), -np.inf, dtype=torch.float64, device=dev)
    state = [(torch.zeros_like(v), torch.zeros_like(v)) for v in params]
    for k in range(1, case["steps"] + 1):
        lb, _, g = step()
        best = torch.maximum(best, lb)
        _adam(params, g, state, k, (0.1, 0.05, 0.05), 1e-8, 1e-3 if E else 0.0)
    lb, _ = last()
    return np.maximum(best.cpu().numpy(), lb), lb


def _inter(net, case, lo, hi, l, u):
    """Optimised intermediate bounds: per (node, side) one set of slopes shared by the rows of a
    layer, ascended on the sum of their bounds; every row keeps its best iterate."""
    l, u = l.clone(), u.clone()
    for t in range(2, net.R + 1):
        d, o = net.dims[t - 1], net.off[t - 1]
        lt, ut = l[:, o:o + d], u[:, o:o + d]
        who, j = torch.nonzero((lt < 0) & (ut > 0), as_tuple=True)
        if not who.numel():
            continue
        best = []
        for sign in (1.0, -1.0):
            rows = torch.zeros(who.numel(), d, dtype=torch.float64, device=lo.device)
            rows[torch.arange(who.numel()), j] = sign
            al = (u >= -l).double()
            state = [(torch.zeros_like(al), torch.zeros_like(al))]
            top = torch.full((who.numel(),), -np.inf, dtype=torch.float64, device=lo.device)
            for k in range(1, case["steps"] + 2):
                p = al.detach().requires_grad_(True)
                v, _ = net.sweep(t, rows, lo[who], hi[who], l[who], u[who], p[who])
                top = torch.maximum(top, v.detach())
                if k > case["steps"]:
                    break
                g, = torch.autograd.grad(v.sum(), [p])
                _adam([al], [g], state, k, (0.1,), 1e-8, 0.0)
            best.append(top)
        lt[who, j] = torch.maximum(lt[who, j], best[0])
        ut[who, j] = torch.minimum(ut[who, j], -best[1])
    return {"l": l.cpu().numpy(), "u": u.cpu().numpy()}
