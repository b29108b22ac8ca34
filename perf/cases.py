"""The measured workloads of this library: what its users run, through its public entry points.

Four kinds of call cover the framework's main path:

* ``job``    a whole run from |0..0>: create a state, evolve it, read every <Z_v>, release it.
* ``step``   one Floquet step of a state with saturated bonds (kick, three gate layers, BP
             regauge), then every <Z_v>; on the periodic cell the bond entropies too.
* ``sweep``  one BP sweep of such a state, then every <Z_v>: regauge and measure.
* ``solve``  the standalone batched truncation solve on device buffers.

The states are random tensors whose bonds carry the spectrum of an evolved kicked-Ising state,
S_k ~ (1 + k)^-0.8 exp(-k / 90), in the gauge that a regauged state has; the kick angles are drawn from the range in which the
dynamics is neither trivial nor Clifford.  Everything random comes from the seed.

``exact`` evaluates the same calls in complex128 with torch and NumPy alone.
"""
import math

import numpy as np
import torch

import paper_2306_14887_gb300 as tn


# ------------------------------------------------------------------------------------ cases
def listed():
    return [
        # the smallest job: one heavy hexagon at chi = 8 over five steps, a point of a theta
        # sweep; launches, synchronisations and handle creation are all there is
        {"name": "ring12_chi8_job_fp32", "kind": "job", "graph": "ring12", "chi": 8,
         "prec": "fp32", "steps": 5},
        # the 127-qubit layout at a small bond dimension in plain FP32: an ordinary exploratory run
        {"name": "eagle127_chi16_step_fp32", "kind": "step", "graph": "eagle127", "chi": 16,
         "prec": "fp32"},
        # a ragged bond dimension on the 65-qubit layout in split TF32
        {"name": "hex65_chi23_step_tf32x3", "kind": "step", "graph": "hex65", "chi": 23,
         "prec": "tf32x3"},
        # the middle of the chi ladder of the 127-qubit layout, in the mode that keeps FP32
        # accuracy on the tensor cores
        {"name": "eagle127_chi32_step_tf32x3", "kind": "step", "graph": "eagle127", "chi": 32,
         "prec": "tf32x3"},
        # its top in plain FP32: the accuracy reference a user checks the other modes with
        {"name": "eagle127_chi64_step_fp32", "kind": "step", "graph": "eagle127", "chi": 64,
         "prec": "fp32"},
        # many instances of uneven size as one handle, each with its own kick angle
        {"name": "union6_chi16_step_tf32x3", "kind": "step", "graph": "union6", "chi": 16,
         "prec": "tf32x3"},
        # the periodic cell of the infinite lattice at a large bond dimension: few, large tensors;
        # its entropy densities are read as well
        {"name": "cell5_chi128_step_fp32", "kind": "step", "graph": "cell5", "chi": 128,
         "prec": "fp32"},
        # regauge and measure in the fastest mode, at the headline size
        {"name": "eagle127_chi64_sweep_tf32", "kind": "sweep", "graph": "eagle127", "chi": 64,
         "prec": "tf32"},
        # the same with FP32 accuracy, and on a 433-qubit layout at half the bond dimension
        {"name": "eagle127_chi64_sweep_tf32x3", "kind": "sweep", "graph": "eagle127", "chi": 64,
         "prec": "tf32x3"},
        {"name": "hex433_chi32_sweep_tf32", "kind": "sweep", "graph": "hex433", "chi": 32,
         "prec": "tf32"},
        # one colour layer's truncation solves at the headline size, and a few odd-sized ones
        {"name": "solve_chi64_51edges", "kind": "solve", "chi": 64, "edges": 51, "sign": 1},
        {"name": "solve_chi21_7edges", "kind": "solve", "chi": 21, "edges": 7, "sign": -1},
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["job", "step", "step", "sweep", "solve", "solve"])
    if kind == "job":
        # within 2^steps <= chi, where nothing is truncated: the product state's symmetries put
        # exact ties into a truncated spectrum, and either choice is then a right one
        steps = rng.randint(3, 5)
        return {"kind": kind, "graph": rng.choice(["ring12", "eagle27"]),
                "chi": 2 ** steps + rng.randint(0, 8), "prec": rng.choice(["fp32", "tf32x3"]),
                "steps": steps}
    if kind == "step":
        graph, largest = rng.choice([("eagle27", 36), ("hex65", 36), ("eagle127", 32),
                                     ("union6", 20)])
        return {"kind": kind, "graph": graph, "chi": log_int(8, largest),
                "prec": rng.choice(["fp32", "tf32x3"])}
    if kind == "sweep":
        return {"kind": kind, "graph": rng.choice(["hex65", "eagle127", "hex433"]),
                "chi": rng.choice([log_int(8, 48), 32, 64]),
                "prec": rng.choice(["tf32", "tf32", "tf32x3", "bf16x3"])}
    return {"kind": kind, "chi": log_int(5, 64), "edges": log_int(1, 60),
            "sign": rng.choice([1, -1])}


# ----------------------------------------------------------------------------------- graphs
def _heavy_hex(rows, cols):
    """(n, edges, colours) of the heavy-hex layout of `rows` rows of `cols` columns: row 0 lacks
    its last column and the last row its first; a bridge below every fourth column."""
    site, bridge, n = {}, {}, 0
    for r in range(rows):
        for c in range(cols):
            if (r, c) not in ((0, cols - 1), (rows - 1, 0)):
                site[r, c] = n
                n += 1
        if r < rows - 1:
            for c in range(2 * (r % 2), cols, 4):
                bridge[r, c] = n
                n += 1
    found = []
    for r in range(rows):
        row = (0, 1, 2, 1) if r % 2 == 0 else (1, 0, 1, 2)
        found += [(site[r, c], site[r, c + 1], row[c % 4]) for c in range(cols - 1)
                  if (r, c) in site and (r, c + 1) in site]
    for (r, c), b in bridge.items():
        found += [(site[r, c], b, 2), (b, site[r + 1, c], 0)]
    found.sort()
    return n, [(u, w) for u, w, _ in found], [k for _, _, k in found]


def _induced(graph, m):
    _, edges, colours = graph
    keep = [i for i, (u, w) in enumerate(edges) if u < m and w < m]
    return m, [edges[i] for i in keep], [colours[i] for i in keep]


def _union(parts):
    n, edges, colours = 0, [], []
    for m, e, c in parts:
        edges += [(u + n, w + n) for u, w in e]
        colours += c
        n += m
    return n, edges, colours


def _graph(name):
    if name == "ring12":
        return 12, [(i, (i + 1) % 12) for i in range(12)], [i % 2 for i in range(12)]
    if name == "cell5":
        return 5, [(0, 2), (0, 3), (0, 4), (1, 2), (1, 3), (1, 4)], [0, 1, 2, 1, 2, 0]
    if name == "eagle27":
        return _induced(_heavy_hex(7, 15), 27)
    if name == "union6":
        small, mid, large = _graph("eagle27"), _heavy_hex(5, 11), _heavy_hex(7, 15)
        return _union([small, mid, large, small, mid, small])
    rows, cols = {"hex65": (5, 11), "eagle127": (7, 15), "hex433": (13, 27)}[name]
    return _heavy_hex(rows, cols)


def _legs(n, edges):
    legs = [[] for _ in range(n)]
    for e, (u, w) in enumerate(edges):
        legs[u].append(e)
        legs[w].append(e)
    return legs


# ----------------------------------------------------------------------------------- inputs
def _spectrum(chi, rank=None):
    """The bond spectrum of an evolved state, of unit 2-norm, zero past its rank."""
    k = torch.arange(chi, dtype=torch.float64)
    s = (1 + k) ** -0.8 * torch.exp(-k / 90)
    s[min(chi, rank or chi):] = 0
    return s / s.norm()


def _ranks(n, edges, chi):
    """The largest rank each bond can have: a site of free legs r_i has at most 2 prod r_i."""
    legs, rank = _legs(n, edges), [chi] * len(edges)
    while True:
        new = [min([rank[e]] + [2 * math.prod(rank[f] for f in legs[v] if f != e) for v in uw])
               for e, uw in enumerate(edges)]
        if new == rank:
            return rank
        rank = new


def _state_inputs(case, seed):
    """(graph, kick angle per vertex, site tensors in complex64, bond spectra).

    Random site tensors in the gauge that BP regauging and the simple update leave: every leg
    carries the root of its bond's spectrum S, and the messages diag(S) are nearly a BP fixed point.
    Per site the condition on leg a is sum G_a G_a'^* prod_b S_b^2 = delta_aa' over the other legs
    b; rounds of whitening one leg after the other come close to it."""
    n, edges, colours = graph = _graph(case["graph"])
    g = torch.Generator(device="cuda").manual_seed(seed)
    chi, legs = case["chi"], _legs(n, edges)
    rank = _ranks(n, edges, chi)
    spectra = torch.stack([_spectrum(chi, r) for r in rank]).float().cuda()
    tensors = [None] * n
    for degree in (1, 2, 3):
        sites = [v for v in range(n) if len(legs[v]) == degree]
        if not sites:
            continue
        # S of every leg, shaped to multiply the batch [site, p, leg 0, ..]
        along = [spectra[[legs[v][i] for v in sites]].reshape(
            (len(sites), 1) + (1,) * i + (chi,) + (1,) * (degree - 1 - i)) for i in range(degree)]
        t = torch.randn((len(sites), 2) + (chi,) * degree, generator=g, device="cuda",
                        dtype=torch.complex64)
        t[:, 0] *= 1.4  # a polarised qubit
        for i in range(degree):
            t *= along[i] > 0
        for i in list(range(degree)) * 16:
            weighted = t * math.prod([along[j] for j in range(degree) if j != i]) if degree > 1 else t
            a = weighted.movedim(i + 2, 1).reshape(len(sites), chi, -1)
            m = a @ a.conj().transpose(-1, -2)
            m += torch.diag_embed((along[i].reshape(len(sites), chi) == 0).to(m.dtype))
            lower = torch.linalg.cholesky(m + 1e-6 * torch.eye(chi, device="cuda"))
            flat = t.movedim(i + 2, 1).reshape(len(sites), chi, -1)
            flat = torch.linalg.solve_triangular(lower, flat, upper=False)
            t = flat.reshape((len(sites), chi, 2) + (chi,) * (degree - 1)).movedim(1, i + 2)
        for i in range(degree):
            t = t * along[i].sqrt()
        for k, v in enumerate(sites):
            tensors[v] = (t[k] / t[k].norm()).contiguous()
    if case["graph"].startswith("union"):  # an angle of its own for each instance
        sizes = [27, 65, 127, 27, 65, 27]
        theta = np.repeat(np.random.default_rng(seed).uniform(0.4, 1.2, len(sizes)), sizes)
    else:
        theta = np.full(n, np.random.default_rng(seed).uniform(0.4, 1.2))
    return graph, theta, tensors, spectra


def _gram_inputs(case, seed):
    """Open-p environments [edge][side][p][re|im][chi][chi] in FP32 of random two-sided bonds."""
    chi, edges = case["chi"], case["edges"]
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.randn((edges, 2, 2, 4 * chi, chi), generator=g, device="cuda",
                    dtype=torch.complex128)
    x *= _spectrum(chi).cuda().sqrt()
    gram = x.transpose(-1, -2) @ x.conj()
    gram /= torch.linalg.matrix_norm(gram)[..., None, None].amax(dim=2, keepdim=True)
    return torch.stack([gram.real, gram.imag], dim=3).float().contiguous()


def prepare(case, seed):
    if case["kind"] == "job":
        theta = float(np.random.default_rng(seed).uniform(0.4, 1.2))
        return {"case": case, "graph": _graph(case["graph"]), "theta": theta}
    if case["kind"] == "solve":
        gram = _gram_inputs(case, seed)
        spectrum = torch.zeros((case["edges"], case["chi"]), dtype=torch.float64, device="cuda")
        return {"case": case, "gram": gram, "legs": torch.zeros_like(gram), "spectrum": spectrum}
    (n, edges, colours), theta, tensors, spectra = _state_inputs(case, seed)
    state = tn.TNState(n, edges, colours, chi=case["chi"], prec=case["prec"])
    for v, t in enumerate(tensors):
        state.set_site(v, t.cpu().numpy())
    messages = torch.diag_embed(spectra).cpu().numpy()
    for e, (u, w) in enumerate(edges):
        message = messages[e]
        state.set_message(e, u, message)
        state.set_message(e, w, message)
    return {"case": case, "state": state, "theta": theta, "edges": len(edges)}


# -------------------------------------------------------------------------------------- run
def run(state):
    """One pass.  Site tensors and messages are held in 32 bits, so what is read off a state is
    kept in 32 bits too; the truncation solve's spectra are 64-bit results.  The solve's leg
    matrices are fixed only up to a unitary freedom on the new bond: what a program makes of them
    is the pair D_v[p] D_w[q]^T that replaces the bond, and that is returned."""
    case = state["case"]
    if case["kind"] == "job":
        n, edges, colours = state["graph"]
        with tn.TNState(n, edges, colours, chi=case["chi"], prec=case["prec"]) as s:
            s.apply_floquet(state["theta"], case["steps"])
            return s.expect_z_all().astype(np.float32)
    if case["kind"] == "solve":
        gram, legs, spectrum = state["gram"], state["legs"], state["spectrum"]
        tn.truncation_solve(gram.data_ptr(), legs.data_ptr(), spectrum.data_ptr(), case["edges"],
                            case["chi"], sign=case["sign"], solve="refined",
                            stream=torch.cuda.current_stream().cuda_stream)
        d = torch.complex(legs[:, :, :, 0], legs[:, :, :, 1])
        pair = d[:, 0][:, :, None] @ d[:, 1].transpose(-1, -2)[:, None]
        return {"spectrum": spectrum.clone(), "pair": pair}
    s = state["state"]
    if case["kind"] == "sweep":
        s.bp_converge(tol=1e-10, max_iters=1)
        return s.expect_z_all().astype(np.float32)
    if case["graph"].startswith("union"):
        s.apply_floquet_field(state["theta"], 1)
    else:
        s.apply_floquet(state["theta"][0], 1)
    z = s.expect_z_all().astype(np.float32)
    if case["graph"] != "cell5":
        return z
    entropy = np.array([s.entanglement_entropy(e) for e in range(state["edges"])])
    return {"z": z, "entropy": entropy.astype(np.float32)}


# ------------------------------------------------------------------------------------- work
def work(case):
    """Per complex multiply-add 8 flops.  A sweep: for a degree-3 site 16 chi^4 of them (five
    mode products and three closes), 8 chi^3 at degree 2, 2 chi^2 at degree 1.  A gate: the open
    environments and the rebuild of its two sites and the solve's decomposition of a
    2 chi x 2 chi matrix (about 20 n^3 flops); a step takes about SWEEPS sweeps to its fixed
    point."""
    chi = case["chi"]
    svd = 20.0 * 4 * (2 * chi) ** 3
    if case["kind"] == "solve":
        edges = case["edges"]
        return {"bytes": edges * (8 * chi ** 2 * 4 + 8 * chi + 4 * chi ** 2 * 8 + 8 * chi ** 2 * 4),
                "flops": edges * svd}
    n, edges, _ = _graph(case["graph"])
    degree = [len(x) for x in _legs(n, edges)]
    state = sum(2 * 8 * chi ** d for d in degree) + 2 * len(edges) * 8 * chi ** 2
    sweep = 8.0 * sum({1: 2 * chi ** 2, 2: 8 * chi ** 3, 3: 16 * chi ** 4}[d] for d in degree)
    measure = 8.0 * sum(d * 2 * chi ** (d + 1) for d in degree)
    gates = len(edges) * svd + 8.0 * sum(
        d * {1: 4 * chi ** 2, 2: 6 * chi ** 3, 3: 8 * chi ** 4}[d] for d in degree)
    if case["kind"] == "sweep":
        return {"bytes": state, "flops": sweep + measure}
    sweeps = 8
    steps = case.get("steps", 1)
    return {"bytes": 2 * state, "flops": steps * (gates + sweeps * sweep) + measure}


# ------------------------------------------------------------------------------------ exact
class _Exact:
    """The same state and updates in complex128: message passing, BP-gauged simple update, <Z>."""

    FLOOR = {"tf32": 2e-3, "bf16x3": 2e-5, "fp32": 2e-6, "tf32x3": 2e-6}
    CUT = {"tf32": 1e-4}

    def __init__(self, graph, chi, prec):
        self.n, self.edges, self.colours = graph
        self.legs = _legs(self.n, self.edges)
        self.chi, self.floor = chi, self.FLOOR[prec]
        self.cut = self.CUT.get(prec, 1e-6)
        z = dict(dtype=torch.complex128, device="cuda")
        self.T = []
        for legs in self.legs:
            t = torch.zeros((2,) + (chi,) * len(legs), **z)
            t.view(-1)[0] = 1
            self.T.append(t)
        m = torch.zeros((chi, chi), **z)
        m[0, 0] = 1
        self.M = {(v, e): m for e, uw in enumerate(self.edges) for v in uw}  # (source, edge)
        self.S = [torch.zeros(chi, dtype=torch.float64) for _ in self.edges]

    def other(self, e, v):
        u, w = self.edges[e]
        return w if u == v else u

    def absorbed(self, v, skip=None):
        """T_v with the incoming messages contracted into every leg but `skip`."""
        t = self.T[v]
        for i, e in enumerate(self.legs[v]):
            if e != skip:
                t = torch.tensordot(t, self.M[self.other(e, v), e], dims=([i + 1], [0]))
                t = t.movedim(-1, i + 1)
        return t

    def message(self, v, e):
        i = self.legs[v].index(e) + 1
        a = self.absorbed(v, e).movedim(i, 0).reshape(self.chi, -1)
        return a @ self.T[v].movedim(i, 0).reshape(self.chi, -1).conj().T

    def sweep(self):
        new, res = {}, 0.0
        for (v, e), old in self.M.items():
            m = self.message(v, e)
            m = 0.5 * (m + m.conj().T)
            new[v, e] = m / torch.linalg.matrix_norm(m)
            res = torch.maximum(torch.as_tensor(res, device="cuda"),
                                torch.linalg.matrix_norm(new[v, e] - old))
        self.M = new
        return float(res)

    def converge(self, limit=1000):
        prev = math.inf
        for it in range(1, limit + 1):
            r = self.sweep()
            if r < 1e-10 or (r < self.floor and (r < self.floor / 8 or (it > 1 and r >= 0.98 * prev))):
                return
            prev = r

    def environments(self, v, e):
        """sum T[p, .., a, ..] conj(T[p, .., b, ..]) over the messages, for p = 0, 1."""
        i = self.legs[v].index(e) + 1
        a = self.absorbed(v, e).movedim(i, 1).reshape(2, self.chi, -1)
        return a @ self.T[v].movedim(i, 1).reshape(2, self.chi, -1).conj().transpose(-1, -2)

    def gate(self, e):
        u, w = self.edges[e]
        both = torch.stack([self.environments(u, e), self.environments(w, e)]).cpu().numpy()
        s, legs = _truncate(both, 1, self.cut)
        for v, d in ((u, legs[0]), (w, legs[1])):
            i = self.legs[v].index(e) + 1
            d = torch.from_numpy(d).cuda()
            t = self.T[v].movedim(i, -1)
            self.T[v] = torch.stack([t[p] @ d[p] for p in range(2)]).movedim(-1, i)
            self.M[v, e] = torch.diag(torch.from_numpy(s)).to(torch.complex128).cuda()
        self.S[e] = torch.from_numpy(s)

    def step(self, theta):
        for v in range(self.n):
            c, s = math.cos(theta[v] / 2), math.sin(theta[v] / 2)
            t = self.T[v]
            self.T[v] = torch.stack([c * t[0] - 1j * s * t[1], c * t[1] - 1j * s * t[0]])
        for colour in sorted(set(self.colours)):
            for e, c in enumerate(self.colours):
                if c == colour:
                    self.gate(e)
        self.converge()

    def z(self):
        out = []
        for v in range(self.n):
            w = (self.absorbed(v) * self.T[v].conj()).reshape(2, -1).sum(1).real
            out.append((w[0] - w[1]) / (w[0] + w[1]))
        return torch.stack(out).cpu().numpy()


def _truncate(env, sign, cut):
    """The kept spectrum and the leg matrices of exp(sign i pi/4 ZZ) on a bond with the open
    environments env[side][p]: N_p = X_p^T conj(X_p), the singular values of
    sum_a X_v[p, r, a] g(p, q) X_w[q, s, a], and the halves mapped back through X."""
    chi = env.shape[-1]
    lam, vec = np.linalg.eigh(0.5 * (env + env.conj().swapaxes(-1, -2)))
    top = lam.max(axis=(1, 2))[:, None, None]
    root = np.sqrt(np.where(lam > 1e-13 * top, lam, 0.0))
    x = root[..., None] * vec.swapaxes(-1, -2)
    inverse = np.divide(1.0, root, out=np.zeros_like(root), where=root > 0)
    phase = np.exp(sign * 0.25j * np.pi * np.array([[1, -1], [-1, 1]]))
    theta = np.einsum("pra,pq,qsa->prqs", x[0], phase, x[1], optimize=True)
    a, s, b = np.linalg.svd(theta.reshape(2 * chi, 2 * chi))
    s = np.where(s[:chi] > cut * s[0], s[:chi], 0.0)
    s = s / np.linalg.norm(s)
    left = (a[:, :chi] * np.sqrt(s)).reshape(2, chi, chi)
    right = (b[:chi].T * np.sqrt(s)).reshape(2, chi, chi)
    return s, [vec[k].conj() @ (inverse[k][..., None] * half)
               for k, half in enumerate((left, right))]


def exact(case, seed):
    if case["kind"] == "solve":
        gram = _gram_inputs(case, seed).double().cpu().numpy()
        env = gram[:, :, :, 0] + 1j * gram[:, :, :, 1]
        done = [_truncate(e, case["sign"], 1e-6) for e in env]
        pair = [np.einsum("pam,qbm->pqab", *legs, optimize=True) for _, legs in done]
        return {"spectrum": np.stack([s for s, _ in done]), "pair": np.stack(pair)}
    if case["kind"] == "job":
        theta = float(np.random.default_rng(seed).uniform(0.4, 1.2))
        x = _Exact(_graph(case["graph"]), case["chi"], case["prec"])
        for _ in range(case["steps"]):
            x.step([theta] * x.n)
        return x.z()
    graph, theta, tensors, spectra = _state_inputs(case, seed)
    x = _Exact(graph, case["chi"], case["prec"])
    x.T = [t.to(torch.complex128) for t in tensors]
    messages = torch.diag_embed(spectra).to(torch.complex128)
    x.M = {(v, e): messages[e] for v, e in x.M}
    del tensors
    if case["kind"] == "sweep":
        x.sweep()
        return x.z()
    x.step(theta)
    if case["graph"] != "cell5":
        return x.z()
    p = torch.stack(x.S).square()
    return {"z": x.z(), "entropy": -torch.special.xlogy(p, p).sum(1).numpy() / math.log(2)}
