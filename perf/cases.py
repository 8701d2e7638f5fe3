"""The work a user of this framework has it do, as cases that can be timed.

Each case is one call (or one training step) through the package's public
entry points, at the sizes of the workloads the repository names (README,
bench.py, workloads.py, optimize.py) and at odd sizes between them.  `draw`
gives more cases of the same ranges, `exact` the results in plain torch
double precision, computed without this package.
"""
from __future__ import annotations

import itertools
import math

import numpy as np
import torch

import paper_2204_00602_gb300 as pcv
from paper_2204_00602_gb300 import autograd as ag
from paper_2204_00602_gb300 import surrogate as sg

DEV = "cuda"

# The surrogate's mesh (12 modes, 6 photons, 132 phases) and its output set.
MESH_M, MESH_N, SET_SIZE = 12, 6, 512


def listed():
    return [
        # the smallest strong simulation: 56 outputs, one photon in each of three modes (latency)
        {"name": "full_m6_n3", "kind": "distribution", "m": 6, "n": 3, "bunched": False},
        # a mid-sized full distribution at odd sizes, several photons per input mode, probabilities and amplitudes
        {"name": "full_m13_n7", "kind": "distribution", "m": 13, "n": 7, "bunched": True},
        # the headline workload: every output of 10 photons in 20 modes, buffers kept between calls
        {"name": "full_m20_n10", "kind": "distribution", "m": 20, "n": 10, "bunched": False},
        # more photons than the tensor-core products take (n > 10)
        {"name": "full_m12_n12", "kind": "distribution", "m": 12, "n": 12, "bunched": False},
        # a requested set of outputs of the headline interferometer, bunched ones among them
        {"name": "amps_m20_n10", "kind": "amplitudes", "m": 20, "n": 10, "outputs": 4096, "bunched": True},
        # one instance of the large-n sweep (m = n^2, 256 collision-free outputs)
        {"name": "amps_m324_n18", "kind": "amplitudes", "m": 324, "n": 18, "outputs": 256, "bunched": False},
        # uneven circuits in one persistent launch, the plan kept
        {"name": "batched_uneven", "kind": "batched", "circuits": 48, "outputs": 512, "m_lo": 8, "m_hi": 64,
         "n_lo": 4, "n_hi": 16, "shape_seed": 3},
        # one step of the differentiable mesh: distribution of 64 phase sets, squared distance to a target, backward
        # to the phases (well conditioned at random phases, where KL's gradient q / p is not)
        {"name": "mesh_step_b64", "kind": "mesh", "m": 12, "n": 6, "batch": 64},
        # training data of the surrogate: exact log-probabilities of its 512 outputs
        {"name": "log_probs_b2048", "kind": "log_probs", "batch": 2048},
        # exact boson sampling at the size of the paper's Boson-sampling benchmark
        {"name": "sample_m60_n14", "kind": "sample", "m": 60, "n": 14, "count": 16384},
        # photon-number-resolved distribution of a lossy, partially distinguishable source
        {"name": "source_m12_n6", "kind": "source", "m": 12, "n": 6, "eta": 0.9, "V": 0.9},
        # one training step of the surrogate network (features, forward, loss, backward, Adam)
        {"name": "train_b4096", "kind": "train", "batch": 4096},
    ]


def _log_int(rng, lo, hi):
    """A whole number spread over the logarithm of [lo, hi]."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _glynn(m, n, outputs):
    """FP64 operations of `outputs` permanents by Glynn's sum with shared row sums (sizes the draws)."""
    return outputs * 2.0 ** (n - 1) * (8 * (n - 1) + 4)


def draw(rng):
    kind = rng.choice(["distribution", "distribution", "amplitudes", "amplitudes", "batched", "mesh", "log_probs",
                       "sample", "source", "train"])
    while True:
        if kind == "distribution":
            m, n = rng.randint(2, 24), rng.randint(1, 12)
            N = pcv.num_outputs(m, n)
            if N <= 20_030_010 and (n <= 10 or N * 2.0 ** (n - 1) <= 1_352_078 * 2048.0):
                return {"kind": kind, "m": m, "n": n, "bunched": rng.random() < 0.5}
        elif kind == "amplitudes":
            n = rng.randint(3, 20)
            bunched = rng.random() < 0.5
            m = _log_int(rng, max(4, n), n * n if n > 12 and not bunched else 64)
            outputs = _log_int(rng, 1, 20_000)
            if _glynn(m, n, outputs) <= _glynn(324, 18, 256):
                return {"kind": kind, "m": m, "n": n, "outputs": outputs, "bunched": bunched}
        elif kind == "batched":
            n_hi = rng.randint(8, 16)
            return {"kind": kind, "circuits": rng.randint(3, 48), "outputs": _log_int(rng, 17, 512), "m_lo": 8,
                    "m_hi": rng.randint(16, 64), "n_lo": rng.randint(3, 6), "n_hi": n_hi,
                    "shape_seed": rng.randrange(1000)}
        elif kind == "mesh":
            m, n, b = rng.randint(4, 14), rng.randint(2, 7), _log_int(rng, 1, 96)
            if b * pcv.num_outputs(m, n) * 2 ** n * n * n <= 64 * 12376 * 64 * 36:
                return {"kind": kind, "m": m, "n": n, "batch": b}
        elif kind == "log_probs":
            return {"kind": kind, "batch": _log_int(rng, 8, 2048)}
        elif kind == "sample":
            n = rng.randint(2, 16)
            m = rng.randint(max(n, 6), 100)
            count = _log_int(rng, 100, 60_000)
            if count * (n * 2.0 ** n + m * n * n) <= 16384 * (14 * 2.0 ** 14 + 60 * 14 * 14):
                return {"kind": kind, "m": m, "n": n, "count": count}
        elif kind == "source":
            m, n = rng.randint(3, 12), rng.randint(1, 6)
            return {"kind": kind, "m": m, "n": n, "eta": round(rng.uniform(0.3, 1.0), 3),
                    "V": round(rng.uniform(0.0, 1.0), 3)}
        else:
            return {"kind": kind, "batch": 32 * _log_int(rng, 1, 128)}


# ------------------------------------------------------------------ inputs

def _haar(m, g):
    z = g.standard_normal((m, m)) + 1j * g.standard_normal((m, m))
    q, r = np.linalg.qr(z)
    d = np.diagonal(r)
    return np.ascontiguousarray(q * (d / np.abs(d))[None, :], dtype=np.complex128)


def _input(m, n, g=None):
    """One photon in each of modes 0..n-1; with a generator, or where there are more photons than
    modes, photons in random modes, several in some."""
    occ = np.zeros(m, dtype=np.uint8)
    if g is None and n <= m:
        occ[:n] = 1
    elif g is None:
        occ[:] = n // m
        occ[:n % m] += 1
    else:
        np.add.at(occ, g.integers(0, m, n), 1)
    return occ


def _outputs(m, n, count, bunched, g):
    """Random outputs: uniform multisets, or uniform n-subsets of the modes."""
    width = m + n - 1 if bunched or n > m else m
    slots = np.sort(np.argsort(g.random((count, width)), axis=1)[:, :n], axis=1)
    modes = slots - np.arange(n)[None, :] if width != m or bunched else slots
    occ = np.zeros((count, m), dtype=np.uint8)
    np.add.at(occ, (np.repeat(np.arange(count), n), modes.reshape(-1)), 1)
    return occ


def _shapes(case):
    g = np.random.default_rng(case["shape_seed"])
    out = []
    for _ in range(case["circuits"]):
        m = int(g.integers(case["m_lo"], case["m_hi"] + 1))
        out.append((m, int(g.integers(case["n_lo"], min(case["n_hi"], m) + 1))))
    return out


def _host(case, seed):
    """The inputs on the host, from the seed alone."""
    g = np.random.default_rng([seed, 20220400])
    kind = case["kind"]
    if kind == "distribution":
        return {"U": _haar(case["m"], g), "t": _input(case["m"], case["n"], g if case["bunched"] else None)}
    if kind == "amplitudes":
        U = _haar(case["m"], g)
        return {"U": U, "t": _input(case["m"], case["n"]),
                "outs": _outputs(case["m"], case["n"], case["outputs"], case["bunched"], g)}
    if kind == "batched":
        return {"circuits": [(_haar(m, g), _input(m, n), _outputs(m, n, case["outputs"], False, g))
                             for m, n in _shapes(case)]}
    if kind == "mesh":
        m, n, B = case["m"], case["n"], case["batch"]
        return {"phases": g.uniform(0, 2 * np.pi, (B, m * (m - 1))), "t": _input(m, n),
                "q": g.dirichlet(np.ones(math.comb(m + n - 1, n)))}
    if kind == "log_probs":
        lists = np.fromiter(itertools.chain.from_iterable(
            itertools.combinations_with_replacement(range(MESH_M), MESH_N)), dtype=np.int64).reshape(-1, MESH_N)
        pick = lists[np.sort(g.choice(len(lists), SET_SIZE, replace=False))]
        outs = np.zeros((SET_SIZE, MESH_M), dtype=np.uint8)
        np.add.at(outs, (np.repeat(np.arange(SET_SIZE), MESH_N), pick.reshape(-1)), 1)
        return {"phases": g.uniform(0, 2 * np.pi, (case["batch"], MESH_M * (MESH_M - 1))),
                "t": _input(MESH_M, MESH_N), "outs": outs}
    if kind == "sample":
        U = _haar(case["m"], g)
        perm = np.argsort(g.random((case["count"], case["n"])), axis=1).astype(np.uint8)
        return {"U": U, "t": _input(case["m"], case["n"]), "perm": perm, "uni": g.random((case["count"], case["n"]))}
    if kind == "source":
        return {"U": _haar(case["m"], g), "t": _input(case["m"], case["n"])}
    B = case["batch"]
    Ws, bs = sg.init_weights(int(g.integers(1 << 30)))
    # targets: log-probabilities of outputs, about log(1 / 12,376) with the spread of exponential probabilities
    return {"Ws": Ws, "bs": bs, "phases": g.uniform(0, 2 * np.pi, (B, sg.P_MESH)),
            "y": (np.log(g.exponential(size=(B, SET_SIZE))) - 9.4).astype(np.float32)}


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


def prepare(case, seed):
    h = _host(case, seed)
    kind = case["kind"]
    s = {"kind": kind, "case": case}
    if kind == "distribution":
        s.update(U=_dev(h["U"]), t=h["t"])
        if pcv.num_outputs(case["m"], case["n"]) > 1_000_000:      # large results: buffers kept between calls
            N = pcv.num_outputs(case["m"], case["n"])
            s["out"] = (torch.empty(N, dtype=torch.float64, device=DEV),
                        torch.empty(N, dtype=torch.complex128, device=DEV))
            s["ws"] = pcv.workspace(pcv.distribution_workspace_bytes(case["m"], case["n"]), s["U"].device)
    elif kind == "amplitudes":
        s.update(U=_dev(h["U"]), t=h["t"], outs=_dev(h["outs"]))
    elif kind == "batched":
        s["plan"] = pcv.BatchPlan([(_dev(U), t, _dev(o)) for U, t, o in h["circuits"]])
    elif kind == "mesh":
        s.update(phases=_dev(h["phases"]).requires_grad_(True), t=h["t"], q=_dev(h["q"]))
    elif kind == "log_probs":
        s.update(phases=_dev(h["phases"]), t=h["t"], outs=_dev(h["outs"]))
    elif kind == "sample":
        s.update(U=_dev(h["U"]), t=h["t"], perm=_dev(h["perm"]), uni=_dev(h["uni"]))
    elif kind == "source":
        s.update(U=_dev(h["U"]), t=h["t"])
    else:
        s.update(net=sg.MLP(h["Ws"], h["bs"], DEV), phases=_dev(h["phases"]), y=_dev(h["y"]))
    return s


def run(s):
    kind, case = s["kind"], s["case"]
    if kind == "distribution":
        return pcv.distribution(s["U"], s["t"], ws=s.get("ws"), out=s.get("out"))
    if kind == "amplitudes":
        return pcv.amplitudes(s["U"], s["t"], s["outs"])
    if kind == "batched":
        amps, probs = s["plan"].run()
        return torch.cat(amps), torch.cat(probs)
    if kind == "mesh":
        s["phases"].grad = None
        p = ag.mesh_distribution(s["phases"], case["m"], s["t"])
        ((p - s["q"]) ** 2).sum().backward()
        return p.detach(), s["phases"].grad
    if kind == "log_probs":
        return sg.exact_log_probs(s["phases"], MESH_M, s["t"], s["outs"])
    if kind == "sample":
        return pcv.sample(s["U"], s["t"], s["perm"], s["uni"])
    if kind == "source":
        return pcv.source_distribution(s["U"], s["t"], case["eta"], case["V"])[0]
    net = s["net"]
    loss = net.train_step(net.features(s["phases"]), s["y"])
    return {"loss": loss, "gW": net.gW, "gb": net.gb}


# -------------------------------------------------------------------- work

def _expansion_flops(m, n):
    """Photon-by-photon expansion over S_{m,1}, ..., S_{m,n}: a complex multiply-add (8 operations) per
    state and occupied mode; m C(m+k-2, k-1) of them at level k."""
    return 8.0 * sum(m * math.comb(m + k - 2, k - 1) for k in range(1, n + 1))


def _amp_flops(m, n, outputs):
    """The fewer of Glynn's sum per output and the expansion of every output."""
    every = _expansion_flops(m, n) if m < 200 else math.inf
    return min(_glynn(m, n, outputs), every)


def work(case):
    kind = case["kind"]
    if kind == "distribution":
        m, n = case["m"], case["n"]
        N = math.comb(m + n - 1, n)
        return {"bytes": 16.0 * m * m + 24.0 * N, "flops": _expansion_flops(m, n) + 3.0 * N}
    if kind == "amplitudes":
        m, n, c = case["m"], case["n"], case["outputs"]
        return {"bytes": 16.0 * m * m + c * (m + 24.0), "flops": _amp_flops(m, n, c)}
    if kind == "batched":
        c = case["outputs"]
        return {"bytes": sum(16.0 * m * m + c * (m + 24.0) for m, n in _shapes(case)),
                "flops": sum(_amp_flops(m, n, c) for m, n in _shapes(case))}
    if kind == "mesh":
        m, n, B = case["m"], case["n"], case["batch"]
        N = math.comb(m + n - 1, n)
        # forward, and two products of the same size in the reverse sweep
        return {"bytes": 16.0 * B * m * (m - 1) + 8.0 * N * (B + 1), "flops": B * (3 * _expansion_flops(m, n) + 10.0 * N)}
    if kind == "log_probs":
        B = case["batch"]
        return {"bytes": 8.0 * B * MESH_M * (MESH_M - 1) + SET_SIZE * (MESH_M + 4.0 * B),
                "flops": B * _amp_flops(MESH_M, MESH_N, SET_SIZE)}
    if kind == "sample":
        m, n, c = case["m"], case["n"], case["count"]
        # per sample n 2^(n-1) complex multiply-adds for the sub-permanents, m n^2 / 2 for the weights
        return {"bytes": 16.0 * m * m + c * (9.0 * n + m), "flops": 8.0 * c * (n * 2.0 ** (n - 1) + m * n * n / 2)}
    if kind == "source":
        m, n = case["m"], case["n"]
        sets = sum(math.comb(n, k) * m * math.comb(m + k - 2, k - 1) for k in range(1, n + 1))
        return {"bytes": 16.0 * m * m + 8.0 * sum(math.comb(m + k - 1, k) for k in range(n + 1)),
                "flops": 8.0 * sets + 2.0 * sum(2 ** (n - j) * m * math.comb(m + j - 1, j) for j in range(1, n + 1))}
    B = case["batch"]
    params = sum(i * o for i, o in zip(sg.DIMS[:-1], sg.DIMS[1:]))
    back = params - sg.DIMS[0] * sg.DIMS[1]
    return {"bytes": 24.0 * params + 8.0 * B * sg.P_MESH + 4.0 * B * SET_SIZE, "flops": 2.0 * B * (2 * params + back)}


# -------------------------------------------------- double precision results

def _counts(m, n):
    """C[w][k]: multisets of size k over w modes."""
    return [[math.comb(w + k - 1, k) if w > 0 else int(k == 0) for k in range(n + 1)] for w in range(m + 1)]


class _Space:
    """The states of S_{m,0}, ..., S_{m,n} in lexicographic order of their sorted mode lists, and for
    each level the rank of every state with one photon taken out of its p-th position."""

    def __init__(self, m, n):
        C = _counts(m, n)
        cum = torch.tensor([[sum(C[m - v][k] for v in range(a)) for a in range(m + 1)] for k in range(n + 1)],
                           device=DEV)
        lists = torch.zeros(1, 0, dtype=torch.int32, device=DEV)
        self.levels, self.m = [], m
        for k in range(1, n + 1):
            last = lists[:, -1].long() if k > 1 else torch.zeros(1, dtype=torch.long, device=DEV)
            cnt = m - last
            idx = torch.repeat_interleave(torch.arange(len(lists), device=DEV), cnt)
            start = torch.cumsum(cnt, 0) - cnt
            new = last[idx] + torch.arange(len(idx), device=DEV) - start[idx]
            lists = torch.cat([lists[idx], new[:, None].int()], 1)
            terms = []
            for p in range(k):
                is_last = torch.ones(len(lists), dtype=torch.bool, device=DEV)
                if p + 1 < k:
                    is_last = lists[:, p] != lists[:, p + 1]
                rank = torch.zeros(len(lists), dtype=torch.long, device=DEV)
                prev = torch.zeros(len(lists), dtype=torch.long, device=DEV)
                pos = 0
                for q in range(k):
                    if q != p:
                        v = lists[:, q].long()
                        rank += cum[k - 2 - pos][v] - cum[k - 2 - pos][prev]
                        prev = v
                        pos += 1
                terms.append((lists[:, p].long(), rank, is_last))
            self.levels.append((lists, terms))

    def norms(self, k):
        """sqrt(prod s!) of the states of level k."""
        if k == 0:
            return torch.ones(1, dtype=torch.float64, device=DEV)
        lists = self.levels[k - 1][0]
        f = torch.ones(len(lists), dtype=torch.float64, device=DEV)
        run = torch.ones_like(f)
        for p in range(1, k):
            run = torch.where(lists[:, p] == lists[:, p - 1], run + 1, torch.ones_like(run))
            f = f * run
        return f.sqrt()

    def amplitudes(self, U, cols):
        """a(S) over S_{m,n} for U [..., m, m] and n photons entering modes `cols`."""
        c = torch.ones(U.shape[:-2] + (1,), dtype=torch.complex128, device=DEV)
        for k in range(1, len(cols) + 1):
            lists, terms = self.levels[k - 1]
            col = U[..., :, cols[k - 1]]
            nxt = 0
            for r, rank, keep in terms:
                nxt = nxt + col[..., r] * c[..., rank] * keep
            c = nxt
        t = np.unique(np.asarray(cols), return_counts=True)[1]
        return c * self.norms(len(cols)) / math.sqrt(math.prod(math.factorial(int(x)) for x in t))

    def step(self, w, x, k):
        """One distinguishable photon of mode probabilities w added to a distribution x over S_{m,k-1}."""
        out = 0
        for r, rank, keep in self.levels[k - 1][1]:
            out = out + w[r] * x[rank] * keep
        return out


def _cols(t):
    return np.repeat(np.arange(len(t)), t).tolist()


def _glynn_amps(U, t, outs):
    """Amplitudes of explicit outputs by Glynn's sum over sign vectors of the input photons; U [B, m, m]."""
    cols = _cols(t)
    n = len(cols)
    rows = torch.from_numpy(np.stack([_cols(o) for o in outs])).to(DEV)
    K = 1 << (n - 1)
    B = U.shape[0]
    chunk = max(1, min(K, (1 << 25) // (B * max(len(outs), U.shape[1]))))
    total = torch.zeros(B, len(outs), dtype=torch.complex128, device=DEV)
    bits = torch.arange(n - 1, device=DEV)
    A = U[:, :, cols].transpose(1, 2)
    for k0 in range(0, K, chunk):
        d = 1.0 - 2.0 * ((torch.arange(k0, min(K, k0 + chunk), device=DEV)[:, None] >> bits) & 1).double()
        d = torch.cat([torch.ones(len(d), 1, dtype=torch.float64, device=DEV), d], 1)
        y = d.to(torch.complex128) @ A                       # [B, chunk, m]
        prod = d.prod(1)[None, :, None].to(torch.complex128)
        for i in range(n):
            prod = prod * y[:, :, rows[:, i]]
        total += prod.sum(1)
    norm = np.array([math.prod(math.factorial(int(x)) for x in o) for o in outs], dtype=np.float64)
    norm *= math.prod(math.factorial(int(x)) for x in t)
    return total / K / torch.from_numpy(np.sqrt(norm)).to(DEV)


def _mesh(phases, m):
    """U(phases) of the rectangular mesh: columns of MZIs diag(1, e^{ib}) BS diag(e^{ia}, 1) BS."""
    B = phases.shape[0]
    rows = list(torch.eye(m, dtype=torch.complex128, device=DEV).expand(B, m, m).unbind(1))
    q = 0
    for c in range(m):
        for k in range(c % 2, m - 1, 2):
            e = torch.exp(1j * phases[:, 2 * q])[:, None]
            f = torch.exp(1j * phases[:, 2 * q + 1])[:, None]
            u0, u1 = rows[k], rows[k + 1]
            rows[k] = 0.5 * ((e - 1) * u0 + 1j * (e + 1) * u1)
            rows[k + 1] = 0.5 * f * (1j * (e + 1) * u0 + (1 - e) * u1)
            q += 1
    return torch.stack(rows, 1)


def exact(case, seed):
    h = _host(case, seed)
    kind = case["kind"]
    if kind == "distribution":
        a = _Space(case["m"], case["n"]).amplitudes(_dev(h["U"]), _cols(h["t"]))
        return a.abs() ** 2, a
    if kind == "amplitudes":
        a = _glynn_amps(_dev(h["U"])[None], h["t"], h["outs"])[0]
        return a, a.abs() ** 2
    if kind == "batched":
        a = torch.cat([_glynn_amps(_dev(U)[None], t, o)[0] for U, t, o in h["circuits"]])
        return a, a.abs() ** 2
    if kind == "mesh":
        ph = _dev(h["phases"]).requires_grad_(True)
        p = _Space(case["m"], case["n"]).amplitudes(_mesh(ph, case["m"]), _cols(h["t"])).abs() ** 2
        q = _dev(h["q"])
        ((p - q) ** 2).sum().backward()
        return p.detach(), ph.grad
    if kind == "log_probs":
        return torch.cat([(_glynn_amps(_mesh(_dev(c), MESH_M), h["t"], h["outs"]).abs() ** 2).log()
                          for c in np.array_split(h["phases"], max(1, len(h["phases"]) // 128))])
    if kind == "sample":
        return None
    if kind == "source":
        m, n = case["m"], case["n"]
        U, cols = _dev(h["U"]), _cols(h["t"])
        space = _Space(m, n)
        q = math.sqrt(case["V"])
        absent, noisy, pure = 1 - case["eta"], case["eta"] * (1 - q), case["eta"] * q
        total = [0.0] * (n + 1)
        for mask in range(1 << n):
            inside = [cols[j] for j in range(n) if mask >> j & 1]
            k = len(inside)
            first = space.amplitudes(U, inside).abs() ** 2 if k else torch.ones(1, dtype=torch.float64, device=DEV)
            blocks = {k: pure ** k * first}
            for j in range(n):
                if not mask >> j & 1:
                    w = U[:, cols[j]].abs() ** 2
                    nxt = {}
                    for b, x in blocks.items():
                        nxt[b] = nxt.get(b, 0.0) + absent * x
                        nxt[b + 1] = nxt.get(b + 1, 0.0) + noisy * space.step(w, x, b + 1)
                    blocks = nxt
            for b, x in blocks.items():
                total[b] = total[b] + x
        zeros = [torch.zeros(math.comb(m + k - 1, k), dtype=torch.float64, device=DEV) for k in range(n + 1)]
        return torch.cat([z + x for z, x in zip(zeros, total)])
    # the training step's loss and gradients; weights and activations unrounded
    ph = _dev(h["phases"])
    X = torch.zeros(len(ph), sg.IN_PAD, dtype=torch.float64, device=DEV)
    P = sg.P_MESH
    X[:, :P], X[:, P:2 * P], X[:, 2 * P] = ph.sin(), ph.cos(), 1.0
    Ws = [_dev(w).double().requires_grad_(True) for w in h["Ws"]]
    bs = [_dev(b).double().requires_grad_(True) for b in h["bs"]]
    x = X
    for i, (w, b) in enumerate(zip(Ws, bs)):
        x = x @ w.T + b
        if i + 1 < len(Ws):
            x = torch.nn.functional.gelu(x)
    loss = ((x - _dev(h["y"]).double()) ** 2).mean()
    loss.backward()
    return {"loss": loss.detach()[None], "gW": [w.grad for w in Ws], "gb": [b.grad for b in bs]}
