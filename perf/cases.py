"""The measured cases: what programs have this library do, over the range of its networks and options.

Every case extracts the polyhedral complex of seeded ReLU networks through
the package's public calls.  Result arrays are read where a program reads
them: on the host (``vertices()`` ...) for the smallest result and from the
server, on the device (``device_arrays()``) for the others, which go on to
further GPU work.  Vertex and edge numbering of the default options varies
from run to run; such a pass ends by putting the arrays into one order with a
few torch calls (by a hash of the packed sign words, which are unique per
vertex), so that they can be matched with another run's.  With
``canonical`` the library fixes the order itself.

A case names its networks (``weights``: the seed that they are drawn from, or
the stored torus net); the seed of ``prepare`` writes the same functions in
another form: the neurons in another order, and another unit of length (a
power of two, so exactly) for the first layer and the box.  Coordinates, sign
vectors and numbering are other ones, and the numbers of cells stay.
"""
import math

import numpy as np
import torch

from paper_2306_07212_gb300 import Extractor, workloads
from paper_2306_07212_gb300.autograd import extract_vertices
from paper_2306_07212_gb300.binding import Server

#: share c of c^D N^D / D! vertices that a net's complex has on [-1, 1]^D, by how its weights are drawn
SHARE = {"he": 0.85, "uniform": 0.45, "torus": 0.48}
#: most vertices a drawn extraction is expected to have (the largest listed one has 1e7)
MOST_VERTICES = 4e6


def expected_vertices(kind, D, width, depth):
    return (SHARE[kind] * (width * depth + 1)) ** D / math.factorial(D) + 2 ** D


def _case(name, net, D, width, depth, precision="mixed", call="extract", order="device", **more):
    c = {"net": net, "weights": 0, "D": D, "width": width, "depth": depth, "precision": precision, "call": call, "order": order,
         "half": 1.0, "prune": False, "vertices": expected_vertices(net, D, width, depth)}
    c.update(more)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest call: a 2-D net of 17 neurons, a few hundred cells, read back to the host for a figure
        _case("small_2d_fp64", "he", 2, 8, 2, "fp64", order="host"),
        # an ordinary point of a counting sweep (four hidden layers), a fixed order so that runs compare
        _case("sweep_2d_w40", "uniform", 2, 40, 4, order="canonical"),
        # the widest layers a served request has, in the plane: few cells, many neuron steps
        _case("wide_2d_w128", "he", 2, 128, 4),
        # the surface network: the SDF of a torus, 3e5 vertices and 9e5 edges, in the default options
        _case("torus_3d", "torus", 3, 64, 4),
        # the same in double precision, in a fixed order
        _case("torus_3d_fp64", "torus", 3, 64, 4, "fp64", order="canonical"),
        # the same network's level set alone, for a mesh
        _case("torus_3d_level_set", "torus", 3, 64, 4, "fp64", prune=True),
        # a window into a wide 4-D net (128-wide layers take the largest tensor-core tiles)
        _case("window_4d_w128", "he", 4, 128, 3, half=0.02, vertices=212e3),
        # the largest: 1e7 vertices, 5e7 edges
        _case("sweep_5d_w40", "uniform", 5, 40, 4, vertices=1.01e7),
        # many dimensions and narrow layers, where every edge has many 2-faces
        _case("sweep_8d_w10", "uniform", 8, 10, 4),
        # a simplex domain and the numbers of its faces of every dimension
        _case("simplex_4d_cells", "uniform", 4, 40, 4, call="cells", order="canonical", vertices=4e4),
        # a training step: the level-set vertices' distance to a sphere, and its gradient
        _case("gradient_3d_w32", "he", 3, 32, 3, "fp64", call="gradient"),
        # small requests of a served stream, eight at a time, results kept on the host
        _case("serve_16", "he", 4, 128, 6, call="serve", requests=16, vertices=16 * 15e3, most=60e3),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["extract"] * 6 + ["level_set", "cells", "gradient", "serve"])
    if call == "serve":
        most = 10 ** rng.uniform(3.5, 4.8)
        n = rng.randint(6, 20)
        return _case(None, "he", 4, 128, 6, call="serve", requests=n, most=most, vertices=0.25 * n * most,
                     weights=rng.randrange(1 << 20))
    for _ in range(1000):
        precision = rng.choice(["mixed", "mixed", "mixed", "fp64"])
        order = rng.choice(["device", "device", "canonical"])
        if call == "cells":
            D = rng.randint(2, 5)
            c = _case(None, "uniform", D, _log(rng, 6, 40), rng.randint(2, 4), precision, "cells", "canonical")
            c["vertices"] /= math.factorial(D)  # the simplex's share of the box
        elif call == "gradient":
            c = _case(None, "he", rng.choice([2, 3]), _log(rng, 8, 48), rng.randint(2, 4), "fp64", "gradient")
        elif call == "level_set":
            c = _case(None, rng.choice(["he", "uniform"]), rng.choice([2, 3]), _log(rng, 10, 64), rng.randint(2, 4),
                      "fp64", order=order, prune=True)
        elif rng.random() < 0.5:
            c = _case(None, "he", rng.choice([2, 3, 4]), _log(rng, 16, 128), rng.randint(2, 6), precision, order=order)
        else:
            c = _case(None, "uniform", rng.randint(1, 8), _log(rng, 10, 40), 4, precision, order=order)
        c["weights"] = rng.randrange(1 << 20)
        most = MOST_VERTICES if call == "extract" and order == "device" else 4e5
        if 100 < c["vertices"] <= most and c["D"] <= c["width"] and (call not in ("gradient", "level_set") or _crosses(c)):
            return c
    raise RuntimeError("no case drawn")


def _crosses(case):
    """Whether the net's output changes its sign in the box (else its level set is empty)."""
    net, box = _inputs(case, 0)
    a = np.random.default_rng(0).uniform(box.lo, box.hi, (500, net.D))
    for W, b in zip(net.W, net.b):
        z = a @ W.T + b
        a = np.maximum(z, 0.0)
    return 25 < int((z > 0).sum()) < 475


# -- inputs ---------------------------------------------------------------------------------------

def _same_function(net, rng):
    """The network with the neurons of each hidden layer in another order, and another unit of length (exact)."""
    W, b = [w.copy() for w in net.W], [v.copy() for v in net.b]
    unit = 2.0 ** int(rng.integers(-3, 4))
    W[0] = W[0] / unit
    for l in range(net.L - 1):
        order = rng.permutation(len(b[l]))
        W[l], b[l], W[l + 1] = W[l][order], b[l][order], W[l + 1][:, order]
    return workloads.Net(list(net.widths), W, b), unit


def _inputs(case, seed):
    """The net and the box (or the simplex) of a case."""
    D = case["D"]
    rng = np.random.default_rng(seed)
    widths = [D] + [case["width"]] * case["depth"] + [1]
    init = workloads.he_normal_mlp if case["net"] == "he" else workloads.default_uniform_mlp
    net = workloads.torus_d3()[0] if case["net"] == "torus" else init(widths, seed=case["weights"]).rounded_to_fp32()
    net, unit = _same_function(net, rng)
    if case["call"] == "cells":
        return net, workloads.Polytope.simplex(D, -unit, 2.0 * unit)
    return net, workloads.Box.cube(D, case["half"] * unit)


def _requests(case, seed):
    """The requests of a served stream (D 2 to 4, depth 2 to 6, width 16 to 128) up to a size."""
    pick, rng = np.random.default_rng(case["weights"]), np.random.default_rng(seed)
    got = []
    while len(got) < case["requests"]:
        D, depth, width = int(pick.integers(2, 5)), int(pick.integers(2, 7)), int(pick.choice([16, 32, 64, 128]))
        if expected_vertices("he", D, width, depth) <= case["most"]:
            net, _ = workloads.random_mlp(D, depth, width, seed=int(pick.integers(1 << 30)))
            net, unit = _same_function(net.rounded_to_fp32(), rng)
            got.append((net, workloads.Box.cube(D, unit)))
    return got


def prepare(case, seed):
    if case["call"] == "serve":
        return {"case": case, "server": Server(max_slots=8, keep_outputs=True), "requests": _requests(case, seed)}
    net, domain = _inputs(case, seed)
    ex = Extractor(precision=case["precision"], canonical=case["order"] != "device" and case["call"] != "gradient",
                   prune=case["prune"], keep_tape=case["call"] == "gradient")
    params = torch.tensor(net.flat_params(), dtype=torch.float64, device="cuda")
    return {"case": case, "ex": ex, "net": net, "domain": domain, "params": params}


# -- one pass -------------------------------------------------------------------------------------

_COEF = np.random.default_rng(7).integers(-2 ** 63, 2 ** 63, 64, dtype=np.int64) | 1
_coef = {}


class _View:
    def __init__(self, ex, ptr, shape, strides, kind):
        self.ex = ex  # owns the memory
        self.__cuda_array_interface__ = {"data": (ptr, False), "shape": shape, "strides": strides, "typestr": kind,
                                         "version": 2}


def _device_views(ex):
    """The context's result arrays: X (D, nV) float64, E (2, nE) int32, sign words (S, nV) as int64."""
    c = ex.counts()
    (px, lx), (pe, le), (ps, ls) = ex.device_arrays()
    X = torch.as_tensor(_View(ex, px, (c["D"], c["nV"]), (8 * lx, 8), "<f8"), device="cuda")
    E = torch.as_tensor(_View(ex, pe, (2, c["nE"]), (4 * le, 4), "<i4"), device="cuda")
    S = torch.as_tensor(_View(ex, ps, (c["S"], c["nV"]), (8 * ls, 8), "<i8"), device="cuda")
    return X, E, S


def _in_order(X, E, S):
    """The same complex, vertices by the hash of their sign words and edges as sorted smaller * nV + larger."""
    nV = X.shape[1]
    if "c" not in _coef:
        _coef["c"] = torch.from_numpy(_COEF).cuda()
    perm = torch.argsort(((S ^ (S >> 23) ^ (S >> 47)) * _coef["c"][: S.shape[0], None]).sum(0))
    rank = torch.empty_like(perm)
    rank[perm] = torch.arange(nV, device=perm.device)
    a, b = rank[E[0]], rank[E[1]]
    edges = torch.sort(torch.minimum(a, b) * nV + torch.maximum(a, b))[0]
    return [X[:, perm], edges, S[:, perm]]


def run(state):
    case = state["case"]
    if case["call"] == "serve":
        srv = state["server"]
        ids = [srv.submit(net, box) for net, box in state["requests"]]
        srv.wait_all()
        out = []
        for rid in ids:
            X, S, E = srv.outputs(rid)
            X, E, S = (torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (X.T, E.T, S.view(np.int64)))
            out += _in_order(X, E, S)
        return out
    ex, net, domain, params = state["ex"], state["net"], state["domain"], state["params"]
    if case["call"] == "gradient":
        theta = params.requires_grad_(True)
        X = extract_vertices(theta, ex, net, domain)
        c = ex.counts()
        word = _device_views(ex)[2][(c["P"] - 1) // 32]
        on = ((word >> (2 * ((c["P"] - 1) % 32))) & 3) == 0  # on the output neuron's zero set
        r = X.norm(dim=1)
        loss = torch.where(on, (r - 1.0) ** 2, torch.zeros_like(r)).sum()
        return [loss.detach(), torch.autograd.grad(loss, theta)[0]]
    if case["call"] == "cells":
        ex.extract_domain(net, domain, params=params)
        f, chi = ex.cell_counts()
        return list(_device_views(ex)) + [f, chi]
    ex.extract(net, domain, params=params)
    if case["order"] == "host":
        return [ex.vertices().T, ex.edges().T, ex.sign_words().view(np.int64)]
    views = _device_views(ex)
    return list(views) if case["order"] == "canonical" else _in_order(*views)


def work(case):
    """Parameters in, coordinates, edges and sign words out; per layer the product over the vertices there at
    its start, and per vertex its interpolation."""
    D, w, depth, V = case["D"], case["width"], case["depth"], case["vertices"]
    if case["call"] == "serve":  # typical requests: D = 3, 64-wide layers
        D, w, depth = 3, 64, 4
    kept = 0.08 * V if case["prune"] else V
    S = (2 * D + w * depth + 1 + 31) // 32
    nparams = w * (D + 1) + (depth - 1) * w * (w + 1) + w + 1
    flops = 0.0
    for l in range(1, depth + 1):
        flops += 2.0 * V * (l / depth) ** D * w * (w if l < depth else 1)
    flops += 4.0 * V * (w + D)
    if case["call"] == "gradient":
        return {"bytes": 24.0 * nparams + V * (16.0 * D + 8 * w), "flops": 3 * flops}
    return {"bytes": 8.0 * nparams + kept * (8.0 * D + 8.0 * S + 8.0 * 0.95 * D), "flops": flops}


# -- the same in 64 bits, by numpy ------------------------------------------------------------------

def exact(case, seed):
    if case["call"] == "serve" or case["vertices"] > 7e5 or case["vertices"] * case["width"] * case["depth"] > 1e8:
        return None
    net, domain = _inputs(case, seed)
    D = net.D
    if case["call"] == "cells":
        A, c, X, E = -domain.A, domain.c, domain.X0, domain.E0.astype(np.int64)
        codes = (np.abs(X @ A.T + c) > 1e-9).astype(np.int8)
    else:
        A = np.zeros((2 * D, D))
        A[np.arange(0, 2 * D, 2), np.arange(D)], A[np.arange(1, 2 * D, 2), np.arange(D)] = 1.0, -1.0
        k = np.arange(1 << D)
        up = ((k[:, None] >> np.arange(D)) & 1).astype(bool)
        X = np.where(up, domain.hi, domain.lo)
        E = np.array([(i, i | (1 << d)) for d in range(D) for i in k if not (i >> d) & 1])
        codes = np.zeros((1 << D, 2 * D), np.int8)
        codes[:, 0::2], codes[:, 1::2] = up, ~up
    X, E, codes = _subdivide(net, A.shape[0], X, E, codes, case["prune"])
    if case["call"] == "gradient":
        return [*_gradient(net, A, X, codes)]
    words = np.zeros(((codes.shape[1] + 31) // 32, len(X)), np.uint64)
    for j in range(codes.shape[1]):
        words[j // 32] |= (codes[:, j] % 3).astype(np.uint64) << np.uint64(2 * (j % 32))
    if case["order"] == "device":
        with np.errstate(over="ignore"):
            words = words.view(np.int64)
            perm = np.argsort(((words ^ (words >> 23) ^ (words >> 47)) * _COEF[: len(words), None]).sum(0))
    else:
        perm = np.lexsort(words[::-1])
    return [np.ascontiguousarray(X[perm].T), None, None] + ([None, None] if case["call"] == "cells" else [])


def _subdivide(net, m, X, E, codes, prune):
    """Edge subdivision, one neuron after the other: signs, split edges, and new edges between the two new
    vertices of every split 2-face (its key: a random linear hash of its sign vector)."""
    D, n = X.shape[1], len(X)
    coef = np.random.default_rng(3).integers(1, 2 ** 63, m + net.n_neurons, dtype=np.int64)
    codes = np.concatenate([codes, np.zeros((n, net.n_neurons), np.int8)], axis=1)
    e = m
    for l, (W, b) in enumerate(zip(net.W, net.b)):
        H = len(b)
        a = X[:n] if l == 0 else np.where(codes[:n, e - W.shape[1]:e] > 0, Z[:n], 0.0)
        Z = a @ W.T + b
        X, codes = X[:n], codes[:n]
        for i in range(H):
            s = np.sign(Z[:n, i])
            codes[:n, e] = s
            ed = np.flatnonzero(s[E[:, 0]] * s[E[:, 1]] < 0)
            if len(ed):
                while n + len(ed) > len(X):
                    X, Z, codes = (np.concatenate([x, np.zeros_like(x)]) for x in (X, Z, codes))
                p, q = E[ed, 0], E[ed, 1]
                flip = s[p] < 0
                p, q = np.where(flip, q, p), np.where(flip, p, q)
                t = (Z[p, i] / (Z[p, i] - Z[q, i]))[:, None]
                zn = Z[p] + t * (Z[q] - Z[p])
                cn = np.where(codes[p] != 0, codes[p], codes[q])
                cn[:, e:] = 0
                zn[:, :i + 1][cn[:, e - i:e + 1] == 0] = 0.0
                new = n + np.arange(len(ed))
                X[new], Z[new], codes[new] = X[p] + t * (X[q] - X[p]), zn, cn
                n += len(ed)
                E[ed] = np.stack([p, new], 1)
                more = [E, np.stack([q, new], 1)]
                if D > 1:
                    zero = np.nonzero(cn[:, :e] == 0)[1].reshape(len(ed), D - 1)
                    with np.errstate(over="ignore"):
                        h = cn[:, :e].astype(np.int64) @ coef[:e]
                        keys = np.stack([h[:, None] + coef[zero], h[:, None] - coef[zero]])
                    real = np.stack([np.ones_like(zero, bool), zero >= m])
                    owner = np.broadcast_to(new[None, :, None], keys.shape)[real]
                    more.append(owner[np.argsort(keys[real], kind="stable")].reshape(-1, 2))
                E = np.concatenate(more)
            e += 1
        if prune and l + 1 < net.L:  # drop the edges that no later neuron can cross
            a, ahead, k = X[:n], [], m
            for q, (Wq, bq) in enumerate(zip(net.W, net.b)):
                v = a @ Wq.T + bq
                if q > l:
                    ahead.append(v > 0)
                a = np.where(v > 0 if q > l else codes[:n, k:k + len(bq)] > 0, v, 0.0)
                k += len(bq)
            ahead = np.packbits(np.concatenate(ahead, axis=1), axis=1)
            E = E[np.any(ahead[E[:, 0]] != ahead[E[:, 1]], axis=1)]
    X, codes = X[:n], codes[:n]
    if prune:
        used = np.unique(E)
        rank = np.zeros(n, np.int64)
        rank[used] = np.arange(len(used))
        X, codes, E = X[used], codes[used], rank[E]
    return X, E, codes


def _gradient(net, A, X, codes):
    """Loss and gradient: each vertex solves its D zero entries, so dL/dtheta = -lambda . dg/dtheta with
    A^T lambda = dL/dx, by a backward pass through the vertex's own affine piece."""
    m, D = A.shape
    on = codes[:, -1] == 0
    X, codes = X[on], codes[on]
    n = len(X)
    r = np.linalg.norm(X, axis=1)
    gx = 2.0 * ((r - 1.0) / r)[:, None] * X
    acts, J, offs, k = [X], [np.broadcast_to(np.eye(D), (n, D, D))], [], m
    rows = np.empty((n, m + net.n_neurons, D), np.float64)
    rows[:, :m] = A
    for W, b in zip(net.W, net.b):
        H = len(b)
        mask = codes[:, k:k + H] > 0
        Jz = W @ J[-1]
        rows[:, k:k + H] = Jz
        acts.append(np.where(mask, acts[-1] @ W.T + b, 0.0))
        J.append(Jz * mask[:, :, None])
        offs.append(k)
        k += H
    zero = np.nonzero(codes == 0)[1].reshape(n, D)
    lam = np.linalg.solve(np.swapaxes(rows[np.arange(n)[:, None], zero], 1, 2), gx[:, :, None])[:, :, 0]
    full = np.zeros((n, m + net.n_neurons))
    full[np.arange(n)[:, None], zero] = -lam
    zbar, grads = None, []
    for l in range(net.L - 1, -1, -1):
        H = len(net.b[l])
        back = 0.0 if zbar is None else (zbar @ net.W[l + 1]) * (codes[:, offs[l]:offs[l] + H] > 0)
        zbar = full[:, offs[l]:offs[l] + H] + back
        grads.append(np.concatenate([(zbar.T @ acts[l]).ravel(), zbar.sum(0)]))
    return np.sum((r - 1.0) ** 2), np.concatenate(grads[::-1])
