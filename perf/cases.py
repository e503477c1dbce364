"""Measured cases: what a user of this framework has it do, through the
Python binding (paper_2007_07379_gb300.pbits).

Kinds of case:
  gibbs    plain or general-gate Gibbs chains of one circuit (PB_GIBBS) or
           the exact samplers (PB_ELIM, PB_ELIM_CLAMP): sweeps, amplitudes
           with their standard errors, chain words
  noalloc  the run that allocates nothing (short calls)
  batch    many uneven circuits in one persistent launch
  learned  the learned proposal as a run mode (a suffix move, then sweeps)
  train    Adam steps of the proposal network on collected paths
  mlp      the network alone: logits and the gradients of one batch
  shor     column sampling of the period-finding circuit and its peaks
"""
from __future__ import annotations

import numpy as np
import torch

from paper_2007_07379_gb300 import pbits
from paper_2007_07379_gb300 import workloads as W

SAMPLERS = {"gibbs": pbits.PB_GIBBS, "elim": pbits.PB_ELIM, "clamp": pbits.PB_ELIM_CLAMP}


def listed():
    return [
        # the smallest call: a plug-in's short run without an allocator (six
        # qubits, the smallest circuit of the batched workload); latency
        {"name": "noalloc_short", "kind": "noalloc", "n": 6, "d": 8, "circuit": 2000, "chains": 256,
         "sweeps": 32},
        # the tiny workload: 3 qubits, 4 layers, 1024 chains x 1e4 sweeps,
        # 8 amplitudes; long chains of a circuit that does not fill a warp
        {"name": "tiny", "kind": "gibbs", "n": 3, "d": 4, "circuit": 0, "chains": 1024,
         "sweeps": 10_000, "sampler": "gibbs", "bins": 0, "frac_u": 0.0},
        # the mid workload (the benchmark's step): 12 qubits, 20 layers, 4096
        # chains x 1e4 sweeps, the full 4096-amplitude histogram
        {"name": "mid", "kind": "gibbs", "n": 12, "d": 20, "circuit": 1000, "chains": 4096,
         "sweeps": 10_000, "sampler": "gibbs", "bins": 0, "frac_u": 0.0},
        # the mid circuit with 30 % general one-qubit gates: Metropolis
        # acceptance of coupled p-bits and FP64 phase sums
        {"name": "general_mid", "kind": "gibbs", "n": 12, "d": 20, "circuit": 1000, "chains": 4096,
         "sweeps": 2_000, "sampler": "gibbs", "bins": 0, "frac_u": 0.3},
        # the large workload: 24 qubits, 32 layers, 65,536 chains, 64 recorded
        # outputs; many chain groups per SM
        {"name": "large", "kind": "gibbs", "n": 24, "d": 32, "circuit": 4000, "chains": 65_536,
         "sweeps": 1_000, "sampler": "gibbs", "bins": 64, "frac_u": 0.0},
        # i.i.d. paths of the mid circuit from the exact sampler
        {"name": "exact_mid", "kind": "gibbs", "n": 12, "d": 20, "circuit": 1000, "chains": 4096,
         "sweeps": 10_000, "sampler": "elim", "bins": 0, "frac_u": 0.0},
        # the batched workload: 256 uneven circuits (6..20 qubits, 8..40
        # layers, 104,960 chains) in one persistent launch
        {"name": "batched", "kind": "batch", "count": 256, "circuit": 2000, "sweeps": 10_000},
        # the learned workload: a suffix move of 4096 chains before every sweep
        {"name": "learned", "kind": "learned", "n": 16, "d": 24, "circuit": 3000, "chains": 4096,
         "hidden": 256, "sweeps": 200, "mh_every": 1},
        # training of its network: batches of 4096 rows from collected paths
        {"name": "train", "kind": "train", "n": 16, "d": 24, "circuit": 3000, "hidden": 256,
         "rows": 4096, "steps": 100},
        # the network alone at the large workload's size, a ragged batch:
        # logits (fused inference kernel) and gradients
        {"name": "mlp_ragged", "kind": "mlp", "n": 24, "d": 32, "hidden": 256, "rows": 1000},
        # the paper's 27-bit period-finding example: 250 columns of 2^27
        {"name": "shor_27bit", "kind": "shor", "N": 98743069, "a": 10424, "n": 27, "T": 250},
        # its Table 1 case: order 479568, T = 3 r columns of 2^20 (a sort of
        # 1.4 million samples and many samples per output)
        {"name": "shor_table1", "kind": "shor", "N": 961307, "a": 5, "n": 20, "T": 3 * 479568},
    ]


def _log_int(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    kind = rng.choice(["gibbs", "gibbs", "gibbs", "exact", "noalloc", "batch", "learned", "train",
                       "mlp", "shor"])
    circuit = rng.randrange(10_000)
    if kind in ("gibbs", "exact"):
        n, d = rng.randint(3, 24), rng.randint(4, 32)
        chains = _log_int(rng, 32, 65_536)
        bins = 0 if n <= 14 else rng.choice([1, 16, 64])
        frac_u = rng.choice([0.0, 0.0, 0.3])
        sampler = "gibbs" if kind == "gibbs" else rng.choice(["elim", "clamp"])
        if sampler == "clamp":
            bins, frac_u = 1, 0.0
        # at most a tenth of the large workload's p-bit updates
        top = max(20, min(10_000, int(5e9 / (n * d * max(chains, 4096)))))
        return {"kind": "gibbs", "n": n, "d": d, "circuit": circuit, "chains": chains,
                "sweeps": _log_int(rng, 10, top), "sampler": sampler, "bins": bins, "frac_u": frac_u}
    if kind == "noalloc":
        return {"kind": "noalloc", "n": rng.randint(3, 12), "d": rng.randint(4, 20), "circuit": circuit,
                "chains": _log_int(rng, 32, 4096), "sweeps": _log_int(rng, 1, 500)}
    if kind == "batch":
        return {"kind": "batch", "count": _log_int(rng, 2, 256), "circuit": circuit,
                "sweeps": _log_int(rng, 10, 1000)}
    if kind == "learned":
        return {"kind": "learned", "n": rng.randint(5, 24), "d": rng.randint(6, 32), "circuit": circuit,
                "chains": _log_int(rng, 64, 16_384), "hidden": rng.choice([64, 128, 256]),
                "sweeps": rng.randint(4, 60), "mh_every": rng.choice([1, 1, 2, 5])}
    if kind == "train":
        return {"kind": "train", "n": rng.randint(5, 24), "d": rng.randint(6, 32), "circuit": circuit,
                "hidden": rng.choice([64, 128, 256]), "rows": 8 * _log_int(rng, 16, 512),
                "steps": _log_int(rng, 1, 100)}
    if kind == "mlp":
        return {"kind": "mlp", "n": rng.randint(5, 24), "d": rng.randint(6, 32),
                "hidden": rng.choice([64, 128, 256]), "rows": 8 * _log_int(rng, 1, 512)}
    n = rng.randint(10, 25)
    N = rng.randrange((1 << (n - 1)) + 1, 1 << n, 2)
    return {"kind": "shor", "N": N, "a": rng.randrange(2, N), "n": n,
            "T": _log_int(rng, 16, max(32, min(1 << 18, (1 << 37) >> n)))}


def _circuit(c):
    """(gates, J, mats) of a case's circuit."""
    n, d = c["n"], c["d"]
    if c.get("frac_u"):
        g, mats = W.random_general_circuit(n, d, seed=c["circuit"], frac_u=c["frac_u"])
        if not np.any(g[:, 0] == W.U):
            mats = None
    else:
        g, mats = W.random_circuit(n, d, seed=c["circuit"]), None
    return g, W.default_J(n, d, g), mats


def _weights(n, d, hidden, seed):
    """Parameters of a network (fp32, uniform +-1/sqrt(fan_in), small biases;
    rows of W3 past n zero), as a program loads them."""
    r = np.random.default_rng(seed)
    k_in, npad = (n + d + 15) // 16 * 16, (n + 15) // 16 * 16
    p = {}
    for i, (rows, cols, live) in enumerate([(hidden, k_in, hidden), (hidden, hidden, hidden), (npad, hidden, n)]):
        w = r.uniform(-1, 1, (rows, cols)) / np.sqrt(cols)
        b = 0.1 * r.uniform(-1, 1, rows)
        w[live:], b[live:] = 0.0, 0.0
        p[f"W{i + 1}"], p[f"b{i + 1}"] = w.astype(np.float32), b.astype(np.float32)
    return p


def _rows(n, d, k_in, rows, seed):
    """Network inputs [2 s_{j-1} - 1, onehot(j-1), 0...] (bf16) and target
    bits (fp32) of uniform layer words and layers."""
    r = np.random.default_rng(seed)
    prev = r.integers(0, 1 << n, size=rows)
    layer = r.integers(0, d, size=rows)
    x = np.zeros((rows, k_in), dtype=np.float32)
    x[:, :n] = 2.0 * ((prev[:, None] >> np.arange(n)) & 1) - 1.0
    x[np.arange(rows), n + layer] = 1.0
    t = (r.random((rows, n)) < 0.5).astype(np.float32)
    return x, t


def _columns(c, seed):
    return np.random.default_rng(seed).integers(0, 1 << c["n"], size=c["T"], dtype=np.uint32)


def _collect(model, net, chains, seed, n_paths):
    """n_paths valid plain-Gibbs paths (int32 [n_paths, d])."""
    src = pbits.Run([model], [pbits.RunCfg(seed=seed, chains=chains, alphas=np.zeros(1, np.uint32))])
    coll = pbits.Learned(src, net)
    paths = torch.zeros((n_paths, model.d), dtype=torch.int32, device="cuda")
    count = torch.zeros(1, dtype=torch.int64, device="cuda")
    src.sweeps(50)
    while int(count.item()) < n_paths:
        src.sweeps(2)
        coll.collect(paths, count)
    coll.close()
    return paths


def prepare(case, seed):
    kind = case["kind"]
    s = {"kind": kind, "case": case}
    key = 0x5EED + 1_000_003 * seed
    if kind in ("gibbs", "noalloc", "learned", "train"):
        g, J, mats = _circuit(case)
        s["model"] = m = pbits.Model(case["n"], case["d"], g, J, mats=mats)
    if kind == "gibbs":
        alphas = np.arange(case["bins"], dtype=np.uint32) if case["bins"] else None
        s["run"] = pbits.Run([m], [pbits.RunCfg(seed=key, chains=case["chains"], alphas=alphas,
                                                sampler=SAMPLERS[case["sampler"]])])
    elif kind == "noalloc":
        s["cfg"] = pbits.RunCfg(seed=key, chains=case["chains"])
        s["counts"] = torch.zeros((1 << case["n"]) * 8, dtype=torch.int64, device="cuda")
        s["totals"] = torch.zeros(2, dtype=torch.int64, device="cuda")
    elif kind == "batch":
        rng = W.SplitMix64(case["circuit"])
        s["models"], cfgs = [], []
        for i in range(case["count"]):
            n, d = 6 + rng.below(15), 8 + rng.below(33)
            g = W.random_circuit(n, d, seed=case["circuit"] + i)
            s["models"].append(pbits.Model(n, d, g, W.default_J(n, d, g)))
            cfgs.append(pbits.RunCfg(seed=key + i, chains=W.chains_for(n),
                                     alphas=np.arange(64, dtype=np.uint32)))
        s["run"] = pbits.Run(s["models"], cfgs)
    elif kind in ("learned", "train"):
        # a short training run on collected paths, as a program does before
        # it samples with the proposal
        rows = case.get("rows", 1024)
        s["net"] = net = pbits.Mlp(case["n"], case["d"], hidden=case["hidden"],
                                   batch=(max(rows, 1024) + 127) // 128 * 128, seed=seed + 3)
        s["paths"] = paths = _collect(m, net, 4096, key + 100, 20_000)
        if kind == "learned":
            pbits.train_on_paths(net, paths, len(paths), 0, steps=100, rows=1024, lr=2e-3, seed=seed)
            alphas = np.arange(16, dtype=np.uint32)
            s["run"] = pbits.Run([m], [pbits.RunCfg(seed=key, chains=case["chains"], alphas=alphas,
                                                    sampler=pbits.PB_LEARNED, proposal=net,
                                                    mh_every=case["mh_every"])])
        else:
            s["seed"] = seed
    elif kind == "mlp":
        rows = case["rows"]
        s["net"] = net = pbits.Mlp(case["n"], case["d"], hidden=case["hidden"],
                                   batch=(rows + 127) // 128 * 128)
        net.set_params(_weights(case["n"], case["d"], case["hidden"], seed))
        x, t = _rows(case["n"], case["d"], net.k_in, rows, seed)
        s["x"] = torch.from_numpy(x).cuda().to(torch.bfloat16)
        s["target"] = torch.from_numpy(t).cuda()
    elif kind == "shor":
        s["cols"] = _columns(case, seed)
        s["sc"] = pbits.ShorColumns(case["n"], case["T"])
    return s


def run(s):
    kind, c = s["kind"], s["case"]
    if kind == "gibbs":
        s["run"].sweeps(c["sweeps"])
        psi, se = s["run"].amplitudes()
        return {"psi": psi, "se": se, "state": s["run"].get_state().view(np.int32)}
    if kind == "noalloc":
        pbits.gibbs_run_noalloc(s["model"], s["cfg"], c["sweeps"], s["counts"], s["totals"])
        return {"counts": s["counts"], "totals": s["totals"]}
    if kind == "batch":
        s["run"].sweeps(c["sweeps"])
        out = [s["run"].amplitudes(i) for i in range(c["count"])]
        return {"psi": np.stack([p for p, _ in out]), "se": np.stack([e for _, e in out]),
                "state": np.concatenate([s["run"].get_state(i).view(np.int32).reshape(-1)
                                         for i in range(c["count"])])}
    if kind == "learned":
        s["run"].sweeps(c["sweeps"])
        psi, se = s["run"].amplitudes()
        moves, accepted = s["run"].moves()
        return {"psi": psi, "se": se, "moves": moves, "accepted": accepted,
                "state": s["run"].get_state().view(np.int32)}
    if kind == "train":
        losses = pbits.train_on_paths(s["net"], s["paths"], len(s["paths"]), 0, steps=c["steps"],
                                      rows=c["rows"], lr=1e-3, seed=s["seed"])
        return {"losses": losses, "params": s["net"].params()}
    if kind == "mlp":
        logits = s["net"].forward_fused(s["x"])
        loss = s["net"].backward(s["x"], s["target"])
        return {"logits": logits, "loss": loss, "grads": s["net"].grads()}
    s["sc"].run(c["N"], c["a"], s["cols"])
    # the order of a is read off as the number of peaks
    count, _, top = s["sc"].peaks(2.2 / (1 << c["n"]), 0)
    return {"prob": s["sc"].prob, "peaks": count, "max": top}


def work(case):
    """Bytes: chain words in and out, records, weights, inputs and outputs.
    Operations: for the samplers the integer lane operations that the bit-
    sliced method cannot do without (132 issue slots per 32-chain word
    update: two Philox calls with an early stop, comparison, links, record;
    the exact sampler: one call per free output, links and record, about 60);
    2 per multiply-add elsewhere."""
    kind = case["kind"]
    if kind in ("gibbs", "noalloc"):
        words = case["n"] * case["d"] * ((case["chains"] + 31) // 32)
        bins = case.get("bins", 0) or (1 << case["n"])
        per = 132 if case.get("sampler", "gibbs") == "gibbs" else 60
        return {"bytes": 8 * words + 24 * bins, "flops": 32.0 * per * words * case["sweeps"]}
    if kind == "batch":
        rng, words = W.SplitMix64(case["circuit"]), 0
        for _ in range(case["count"]):
            n, d = 6 + rng.below(15), 8 + rng.below(33)
            words += n * d * (W.chains_for(n) // 32)
        return {"bytes": 8 * words + 24 * 64 * case["count"], "flops": 32.0 * 132 * words * case["sweeps"]}
    n, d = case["n"], case.get("d", 0)
    if kind == "shor":
        # one complex multiply-add per (k, sample)
        return {"bytes": 8.0 * (1 << n) + 4 * case["T"], "flops": 8.0 * (1 << n) * case["T"]}
    h, k_in, npad = case["hidden"], (n + d + 15) // 16 * 16, (n + 15) // 16 * 16
    weights = h * (k_in + h + npad)
    if kind == "learned":
        moves = case["sweeps"] // case["mh_every"]
        words = n * d * ((case["chains"] + 31) // 32)
        # a suffix of (d + 1) / 2 layers on average: the draw and log q of both
        return {"bytes": 8 * words + 2 * weights,
                "flops": moves * case["chains"] * (d + 1) * 2.0 * weights +
                32.0 * 132 * words * case["sweeps"]}
    if kind == "train":
        return {"bytes": case["steps"] * (24 * weights + 4 * case["rows"] * 2),
                "flops": case["steps"] * 6.0 * weights * case["rows"]}
    # mlp: logits, then the backward pass with its own forward
    return {"bytes": 6 * weights + case["rows"] * (2 * k_in + 8 * n), "flops": 8.0 * weights * case["rows"]}


def _exact_mlp(case, seed):
    """Logits, binary cross-entropy and its gradients in FP64 from the
    fp32 parameters."""
    n, d = case["n"], case["d"]
    p = _weights(n, d, case["hidden"], seed)
    x, t = _rows(n, d, (n + d + 15) // 16 * 16, case["rows"], seed)
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    q = {k: torch.from_numpy(v).double().to(dev).requires_grad_(True) for k, v in p.items()}
    X, Tt = torch.from_numpy(x).double().to(dev), torch.from_numpy(t).double().to(dev)
    h1 = torch.relu(X @ q["W1"].T + q["b1"])
    h2 = torch.relu(h1 @ q["W2"].T + q["b2"])
    logits = (h2 @ q["W3"].T + q["b3"])[:, :n]
    # summed over a row's bits, mean over the rows
    loss = torch.nn.functional.binary_cross_entropy_with_logits(logits, Tt, reduction="sum") / len(x)
    loss.backward()
    return {"logits": logits.detach(), "loss": loss.detach().reshape(1),
            "grads": {k: v.grad.cpu().numpy() for k, v in q.items()}}


def _exact_shor(case, seed):
    """P[k] = sum_y |sum_{i: y_i = y} e^{2 pi i k x_i / 2^n}|^2 2^-n / T as one
    FFT of the histogram of the differences x_i - x_j within each y."""
    n, N, T = case["n"], case["N"], case["T"]
    x = _columns(case, seed).astype(np.uint64)
    y = np.full(T, 1 % N, dtype=np.uint64)
    b, e = case["a"] % N, x.copy()
    while np.any(e):  # N < 2^32: the products fit 64 bits
        y = np.where(e & np.uint64(1), y * np.uint64(b) % np.uint64(N), y)
        b, e = b * b % N, e >> np.uint64(1)
    order = np.lexsort((x, y))
    x, y = x[order].astype(np.int64), y[order]
    M = 1 << n
    c = np.zeros(M)
    c[0] = T
    s = 1
    while s < T:
        same = y[s:] == y[:-s]
        if not same.any():
            break
        diff = (x[s:] - x[:-s])[same] % M
        np.add.at(c, diff, 1.0)
        np.add.at(c, (M - diff) % M, 1.0)
        s += 1
        if s > 2000:
            return None
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    P = torch.fft.fft(torch.from_numpy(c).to(dev)).real
    P = P * (2.0 ** -n / T)
    return {"prob": P.contiguous(), "peaks": None, "max": float(P.max())}


def exact(case, seed):
    # the samplers' outputs are whole numbers (chain words, counts) and
    # amplitudes formed from them; no 64-bit value of a sampled estimate
    # exists without the sampler itself
    if case["kind"] == "mlp":
        return _exact_mlp(case, seed)
    if case["kind"] == "shor":
        return _exact_shor(case, seed)
    return None
