"""Performance cases of the LABS search library: what its users run, through the public entry points.

A case is a dict of plain values with a ``kind``:

  walk       step 1 of the search (labs_skew_search): self-avoiding walks behind 24-element prefixes, with the
             sieve bound sampled in the call or switched off
  mixed      step 1 over every length of a range in one persistent launch (labs_batched_search, graph replay)
  collect    walks in chunks with their states and moves logged (labs_chunked_search), the learned proposal's
             training data
  pq         step 2 with one shared queue (labs_pq_refine)
  pq_indep   step 2 with one queue per candidate (labs_pq_independent)
  energy     energies (and correlation tables) of a batch of sequences (labs_energy_batch)
  deltas     energy changes of every neighbour of a batch of sequences (labs_flip_deltas)
  operators  the end-element operators between the lengths (labs_sequence_operators)
  forward    the proposal network's logits (Policy.forward)
  train      one training step of the proposal network with its gradients (Policy.train_step)

Energies, sequences and statistics are exact integers; the network's outputs are FP32.
"""
import math

import numpy as np
import torch

import paper_2409_07222_gb300 as lg

INT32_MAX = 2**31 - 1
HIDDEN, CHANNELS, TAPS = 256, 64, 9


def listed():
    return [
        # the headline search: 65,536 walks at L = 451 behind 256 prefixes, bound = 1000th of 10^6 sampled starts;
        # a little more than one walk segment (1808 flips), so restarts are part of it
        dict(name="walk_451", kind="walk", L=451, p=24, n_walks=65536, flips=2000, R=16, samples=10**6, rank=999),
        # one evaluation run of the learned-proposal comparison: few walks, long budget -- latency of one step
        dict(name="walk_451_few", kind="walk", L=451, p=24, n_walks=256, flips=8192, R=4, samples=0, rank=0),
        # a search over the paper's whole range of lengths, odd ones skew-symmetric, even ones unrestricted
        dict(name="mixed_450_527", kind="mixed", L_min=450, L_max=527, p=24, lo=64, hi=1024, flips=500, R=16,
             samples=10**6, rank=999),
        # training data for the proposal network: chunks of 64 flips, state and first move of each logged
        dict(name="collect_451", kind="collect", L=451, p=24, n_walks=2048, flips=1024, chunk=64, R=4),
        # step 2 from the 4,096 best step-1 candidates, as the two-step search runs it
        dict(name="pq_451", kind="pq", L=451, seeds=4096, B=4096, cap=1 << 22, expansions=10**6, T_r=0, H_log2=28),
        # step 2 at the even neighbour length from the few sequences the operators give, rotations on, a queue
        # small enough to evict: rounds are small, so launches and latency count
        dict(name="pq_452_few", kind="pq", L=452, seeds=4, B=256, cap=1 << 16, expansions=20000, T_r=4, H_log2=24),
        # step 2 as the paper parallelises it: one search per candidate
        dict(name="pq_indep_451", kind="pq_indep", L=451, seeds=4096, pops=256, T_r=0, H_log2=18),
        # the sieve sample's shape: energies of a million sequences
        dict(name="energy_451", kind="energy", L=451, n=1 << 20, with_C=False),
        # the neighbour scan alone on a batch of skew-symmetric sequences, tables built in the call
        dict(name="deltas_451", kind="deltas", L=451, n=1 << 15, skew=True, p=24, give_C=False),
        # the smallest call: the operators on step 2's best sequence
        dict(name="operators_one", kind="operators", L=451, n=1),
        # the network scores every walk's state before a chunk
        dict(name="forward_451", kind="forward", L=451, n=8192),
        # one minibatch of the network's training
        dict(name="train_451", kind="train", L=451, p=24, n=512),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _neighbours(L, skew, p):
    return (L + 1) // 2 - p if skew else L - p


def _lags(L, skew):
    return (L - 1) // 2 if skew else L - 1


_LARGEST_WALK = 65536 * 2000 * _neighbours(451, True, 24) * _lags(451, True)  # neighbour-lag terms


def draw(rng):
    kind = rng.choice(["walk", "walk", "mixed", "collect", "pq", "pq_indep", "energy", "energy", "deltas", "deltas",
                       "operators", "forward", "train"])
    L = _log_int(rng, 64, 576)
    p = rng.choice([0, 7, 13, 24])
    if kind == "walk":
        skew = L % 2 == 1
        n = _log_int(rng, 16, 65536)
        room = _LARGEST_WALK // (n * _neighbours(L, skew, p) * _lags(L, skew))
        flips = max(1, min(_log_int(rng, 200, 8192), room))
        samples = rng.choice([0, _log_int(rng, 1000, 10**6)])
        return dict(kind=kind, L=L, p=p, n_walks=n, flips=flips, R=rng.choice([1, 4, 16, 32]), samples=samples,
                    rank=samples // 1000)
    if kind == "mixed":
        L_min = rng.randint(448, 520)
        return dict(kind=kind, L_min=L_min, L_max=min(527, L_min + rng.randint(1, 40)), p=24, lo=16,
                    hi=_log_int(rng, 32, 1024), flips=_log_int(rng, 100, 500), R=rng.choice([4, 16]), samples=10**5,
                    rank=99)
    if kind == "collect":
        return dict(kind=kind, L=L | 1 if L < 576 else 575, p=p, n_walks=_log_int(rng, 64, 2048),
                    flips=_log_int(rng, 64, 1024), chunk=rng.choice([16, 64, 256]), R=4)
    if kind == "pq":
        return dict(kind=kind, L=min(L, 527), seeds=_log_int(rng, 1, 4096), B=rng.choice([64, 256, 1000, 4096]),
                    cap=1 << rng.choice([14, 18, 22]), expansions=_log_int(rng, 2000, 50000),
                    T_r=rng.choice([0, 0, 4]), H_log2=26)
    if kind == "pq_indep":
        return dict(kind=kind, L=min(L, 527), seeds=_log_int(rng, 64, 4096), pops=_log_int(rng, 16, 256),
                    T_r=rng.choice([0, 0, 4]), H_log2=18)
    if kind == "energy":
        with_C = rng.random() < 0.4
        return dict(kind=kind, L=_log_int(rng, 13, 576), n=_log_int(rng, 1, (1 << 20) * 451**2 // 576**2 // (4 if with_C else 1)),
                    with_C=with_C)
    if kind == "deltas":
        skew = rng.random() < 0.5
        L = (L | 1 if L < 576 else 575) if skew else L
        return dict(kind=kind, L=L, n=_log_int(rng, 1, (1 << 15) if skew else (1 << 12)), skew=skew, p=p,
                    give_C=rng.random() < 0.4)
    if kind == "operators":
        return dict(kind=kind, L=min(L, 575), n=_log_int(rng, 1, 1 << 16))
    if kind == "forward":
        return dict(kind=kind, L=min(L, 451), n=_log_int(rng, 1, 8192))
    return dict(kind=kind, L=min(L, 451), p=p, n=_log_int(rng, 16, 512))


# ---- inputs --------------------------------------------------------------------------------------------------------

def _prefixes(p, seed):
    """256 distinct prefixes of p elements (fewer when p is short)."""
    if p == 0:
        return torch.zeros(1, dtype=torch.int64, device="cuda")
    n = min(256, 2**p)
    rng = np.random.default_rng(seed)
    v = rng.choice(2**p, size=n, replace=False) if p < 16 else np.unique(rng.integers(0, 2**p, size=2 * n))[:n]
    return torch.from_numpy(np.ascontiguousarray(rng.permutation(v).astype(np.int64))).cuda()


def _random_words(L, n, seed):
    """n uniform sequences as packed words, int64 [n, ceil(L/64)]."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    W = (L + 63) // 64
    w = torch.randint(-2**63, 2**63 - 1, (n, W), generator=g, device="cuda", dtype=torch.int64)
    tail = L - 64 * (W - 1)
    if tail < 64:
        w[:, W - 1] &= (1 << tail) - 1
    return w


def _pack(bits):
    """bool [n, L] -> int64 words."""
    n, L = bits.shape
    W = (L + 63) // 64
    x = torch.zeros((n, W * 64), dtype=torch.int64, device=bits.device)
    x[:, :L] = bits
    one = torch.ones(64, dtype=torch.int64, device=bits.device) << torch.arange(64, device=bits.device)
    return (x.view(n, W, 64) * one).sum(-1)


def _signs(words, L):
    """int64 words [n, W] -> +-1 float64 [n, L]."""
    sh = torch.arange(64, device=words.device)
    b = (words[:, :, None] >> sh) & 1
    return (2 * b.reshape(words.shape[0], -1)[:, :L] - 1).to(torch.float64)


def _skew_words(L, p, n, seed):
    """Skew-symmetric sequences of odd L: s_{c+j} = (-1)^j s_{c-j}, the first p elements one of the prefixes."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    c = (L - 1) // 2
    b = torch.rand((n, L), generator=g, device="cuda") < 0.5
    if p:
        pre = _prefixes(p, seed)
        pb = (pre[torch.arange(n, device="cuda") % pre.numel(), None] >> torch.arange(p, device="cuda")) & 1
        b[:, :p] = pb.bool()
    j = torch.arange(1, c + 1, device="cuda")
    b[:, c + j] = b[:, c - j] ^ (j % 2 == 1)
    return _pack(b)


def _sieved(L, n, seed):
    """The n best states of a short step-1 search, one per walk: what step 2 starts from."""
    skew, p = L % 2 == 1, (24 if L % 2 == 1 and L > 64 else 0)
    cfg = lg.make_walk_cfg(L, skew=skew, p=p, n_walks=n, flip_budget=300, seed=seed, R=1, E_thr=INT32_MAX)
    out, _, _ = lg.labs_skew_search(cfg, _prefixes(p, seed), with_walk_stats=False)
    rec = out.view(torch.int64).view(n, 12)
    return rec[:, 3:3 + (L + 63) // 64].contiguous()


def _network(L, seed):
    """Flat FP32 parameters: He-uniform weights that BF16 holds exactly, small biases."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    flat = []
    for shape in _shapes(L):
        if len(shape) == 1:
            flat.append(0.05 * torch.randn(shape, generator=g, device="cuda"))
        else:
            lim = math.sqrt(6.0 / math.prod(shape[1:]))
            w = (2 * torch.rand(shape, generator=g, device="cuda") - 1) * lim
            flat.append(w.to(torch.bfloat16).to(torch.float32).reshape(-1))
    return torch.cat(flat)


def _shapes(L):
    c = CHANNELS
    return [(c, 2, TAPS), (c,), (c, c, TAPS), (c,), (c, c, TAPS), (c,), (HIDDEN, c * L), (HIDDEN,), (L, HIDDEN), (L,)]


def _train_batch(case, seed):
    n, L, p = case["n"], case["L"], case["p"]
    lo, hi = p, ((L + 1) // 2 if L % 2 else L) - 1
    g = torch.Generator(device="cuda").manual_seed(seed + 1)
    target = torch.randint(lo, hi + 1, (n,), generator=g, device="cuda", dtype=torch.int32)
    weight = torch.randn(n, generator=g, device="cuda").clamp_min(0.0)
    weight[0] = 1.0
    return _random_words(L, n, seed), target, weight, lo, hi


def _batch_plan(case):
    lengths = list(range(case["L_min"], case["L_max"] + 1))
    walks = np.random.default_rng(2410).integers(case["lo"], case["hi"] + 1, size=len(lengths)).tolist()
    return lengths, walks


def prepare(case, seed):
    kind = case["kind"]
    st = dict(case)
    if kind in ("walk", "collect"):
        st["pre"] = _prefixes(case["p"], seed)
        samples = case.get("samples", 0)
        st["cfg"] = lg.make_walk_cfg(case["L"], skew=case["L"] % 2 == 1, p=case["p"], n_walks=case["n_walks"],
                                     flip_budget=case["flips"], seed=seed, R=case["R"],
                                     E_thr=lg.LABS_AUTO_THRESHOLD if samples else INT32_MAX,
                                     n_thresh_samples=samples, thresh_rank=case.get("rank", 0))
    elif kind == "mixed":
        st["lengths"], st["walks"] = _batch_plan(case)
        st["pre"] = _prefixes(case["p"], seed)
        st["cfg"] = lg.make_batch_cfg(len(st["lengths"]), p=case["p"], flip_budget=case["flips"], seed=seed,
                                      R=case["R"], n_thresh_samples=case["samples"], thresh_rank=case["rank"])
        # a program that searches for hours runs the batch once to have it tuned and captured
        st["out"] = lg.labs_batched_search(st["cfg"], st["lengths"], st["walks"], st["pre"])
    elif kind in ("pq", "pq_indep"):
        st["words"] = _sieved(case["L"], case["seeds"], seed)
    elif kind == "deltas":
        st["words"] = (_skew_words(case["L"], case["p"], case["n"], seed) if case["skew"]
                       else _random_words(case["L"], case["n"], seed))
        st["C"] = lg.labs_energy_batch(st["words"], case["L"], with_C=True)[1] if case["give_C"] else None
    elif kind in ("energy", "operators"):
        st["words"] = _random_words(case["L"], case["n"], seed)
    elif kind in ("forward", "train"):
        st["net"] = lg.Policy(case["L"], seed=1)
        st["net"].set_params(_network(case["L"], seed))
        if kind == "forward":
            st["words"] = _random_words(case["L"], case["n"], seed)
        else:
            st["batch"] = _train_batch(case, seed)
    return st


def run(st):
    kind = st["kind"]
    if kind == "walk":
        return lg.labs_skew_search(st["cfg"], st["pre"])
    if kind == "mixed":
        return lg.labs_batched_search(st["cfg"], st["lengths"], st["walks"], st["pre"], out=st["out"])
    if kind == "collect":
        r = lg.labs_chunked_search(st["cfg"], st["pre"], chunk=st["chunk"], log_states=True, log_moves=True)
        return {k: v for k, v in r.items() if v is not None}
    if kind == "pq":
        return lg.labs_pq_refine(st["L"], st["words"], B=st["B"], cap=st["cap"], H_log2=st["H_log2"],
                                 max_expansions=st["expansions"], T_r=st["T_r"])
    if kind == "pq_indep":
        return lg.labs_pq_independent(st["L"], st["words"], st["pops"], T_r=st["T_r"], H_log2=st["H_log2"])
    if kind == "energy":
        return lg.labs_energy_batch(st["words"], st["L"], with_C=st["with_C"])
    if kind == "deltas":
        return lg.labs_flip_deltas(st["words"], st["L"], skew=st["skew"], p=st["p"], C=st["C"])
    if kind == "operators":
        return lg.labs_sequence_operators(st["L"], st["words"])
    if kind == "forward":
        return st["net"].forward(st["words"])
    words, target, weight, lo, hi = st["batch"]
    return st["net"].train_step(words, target, weight, lo, hi, 1e-3, want_grads=True)


# ---- work ----------------------------------------------------------------------------------------------------------

def _energy_flops(L):
    return L * (L - 1)  # one multiply-add per product of every lag


def _flip_flops(L, skew, p):
    # a flip changes one product pair of every lag and, of every neighbour's energy change, one second difference
    return 8.0 * (_neighbours(L, skew, p) + _lags(L, skew))


def _network_flops(L):
    return 2 * CHANNELS * (2 + 2 * CHANNELS) * TAPS * L + 2 * HIDDEN * CHANNELS * L + 2 * HIDDEN * L


def work(case):
    kind = case["kind"]
    W = lambda L: 8 * ((L + 63) // 64)  # noqa: E731
    if kind == "mixed":
        by = fl = 0.0
        mean = 0.5 * (case["lo"] + case["hi"])
        for L in range(case["L_min"], case["L_max"] + 1):
            skew = L % 2 == 1
            fl += mean * case["flips"] * _flip_flops(L, skew, case["p"] if skew else 0)
            fl += case["samples"] * _energy_flops(L) / (2 if skew else 1)
            by += mean * (96 * case["R"] + 48)
        return {"bytes": by, "flops": fl}
    L = case["L"]
    skew = L % 2 == 1
    if kind in ("walk", "collect"):
        by = case["n_walks"] * (96 * case["R"] + 48.0)
        fl = case["n_walks"] * case["flips"] * _flip_flops(L, skew, case["p"])
        fl += case.get("samples", 0) * _energy_flops(L) / (2 if skew else 1)
        if kind == "collect":
            by += case["n_walks"] * -(-case["flips"] // case["chunk"]) * (W(L) + 8.0)
        return {"bytes": by, "flops": fl}
    if kind in ("pq", "pq_indep"):
        pops = case["expansions"] if kind == "pq" else case["pops"] * case["seeds"]
        # every pop: its neighbours' energy changes from its parent's, and one visited-set word per neighbour
        return {"bytes": case["seeds"] * W(L) + pops * 8.0 * L, "flops": pops * _flip_flops(L, False, 0)}
    if kind == "energy":
        out = 4.0 * (L if case["with_C"] else 1)
        return {"bytes": case["n"] * (W(L) + out), "flops": case["n"] * float(_energy_flops(L))}
    if kind == "deltas":
        n, lags, nb = case["n"], _lags(L, case["skew"]), _neighbours(L, case["skew"], case["p"])
        build = 0 if case["give_C"] else _energy_flops(L) / (2 if case["skew"] else 1)
        return {"bytes": n * (W(L) + 4.0 * L + (4.0 * (L - 1) if case["give_C"] else 0)),
                "flops": n * (2.0 * nb * lags + build)}
    if kind == "operators":
        n = case["n"]
        return {"bytes": n * (W(L) + 4.0 * W(L + 1) + 2 * W(L - 1) + 24),
                "flops": n * (4.0 * _energy_flops(L + 1) + 2 * _energy_flops(L - 1))}
    n_params = sum(math.prod(s) for s in _shapes(L))
    if kind == "forward":
        return {"bytes": case["n"] * (W(L) + 4.0 * L) + 2.0 * n_params, "flops": case["n"] * float(_network_flops(L))}
    # forward, both gradients, the update of parameters and two moments; gradients written
    return {"bytes": case["n"] * (W(L) + 8.0) + 4.0 * n_params * (3 + 3 + 1),
            "flops": case["n"] * 3.0 * _network_flops(L)}


# ---- 64-bit values -------------------------------------------------------------------------------------------------

def _corr(s):
    """C_1..C_{L-1} of +-1 rows, float64 (exact after rounding)."""
    L = s.shape[1]
    m = 1 << (2 * L - 1).bit_length()
    f = torch.fft.rfft(s, n=m)
    return torch.round(torch.fft.irfft(f * f.conj(), n=m)[:, 1:L])


def _energies(s, rows=32768):
    return torch.cat([_corr(s[i:i + rows]).square().sum(1) for i in range(0, s.shape[0], rows)]).to(torch.int32)


def _exact_energy(case, seed):
    words, L = _random_words(case["L"], case["n"], seed), case["L"]
    E, C = [], []
    for i in range(0, words.shape[0], 32768):
        c = _corr(_signs(words[i:i + 32768], L))
        E.append(c.square().sum(1).to(torch.int32))
        if case["with_C"]:
            C.append(c.to(torch.int32))
    return (torch.cat(E), torch.cat(C)) if case["with_C"] else torch.cat(E)


def _exact_deltas(case, seed):
    L, n, skew, p = case["L"], case["n"], case["skew"], case["p"]
    words = _skew_words(L, p, n, seed) if skew else _random_words(L, n, seed)
    s = _signs(words, L)
    E0 = _energies(s)
    dE = torch.full((n, L), INT32_MAX, dtype=torch.int32, device=s.device)
    for m in range(p, (L + 1) // 2 if skew else L):
        t = s.clone()
        t[:, m] = -t[:, m]
        if skew and m != L - 1 - m:
            t[:, L - 1 - m] = -t[:, L - 1 - m]
        dE[:, m] = _energies(t) - E0
    return dE


def _exact_operators(case, seed):
    L = case["L"]
    words = _random_words(L, case["n"], seed)
    s = _signs(words, L)
    one = torch.ones((s.shape[0], 1), dtype=s.dtype, device=s.device)
    grow = [torch.cat(v, 1) for v in ((s, one), (s, -one), (one, s), (-one, s))]
    shrink = [s[:, :-1], s[:, 1:]]
    return (torch.stack([_pack(g > 0) for g in grow], 1), torch.stack([_energies(g) for g in grow], 1),
            torch.stack([_pack(g > 0) for g in shrink], 1), torch.stack([_energies(g) for g in shrink], 1))


def _tensors(flat, L):
    out, o = [], 0
    for shape in _shapes(L):
        k = math.prod(shape)
        out.append(flat[o:o + k].reshape(shape))
        o += k
    return out


def _logits(words, L, flat):
    w1, b1, w2, b2, w3, b3, W4, b4, W5, b5 = _tensors(flat, L)
    s = _signs(words, L)
    k = torch.arange(1, L, device=s.device, dtype=torch.float64)
    x = torch.stack([s, torch.cat([torch.zeros_like(s[:, :1]), _corr(s) / torch.sqrt(L - k)], 1)], 1)
    for w, b in ((w1, b1), (w2, b2), (w3, b3)):
        cols = torch.nn.functional.pad(x, (TAPS // 2, TAPS // 2)).unfold(2, TAPS, 1)  # [n, c, L, taps]
        cols = cols.permute(0, 2, 1, 3).reshape(-1, w.shape[1] * TAPS)
        y = cols @ w.reshape(w.shape[0], -1).T + b
        x = torch.relu(y.reshape(s.shape[0], L, -1).permute(0, 2, 1))
    return torch.relu(x.reshape(s.shape[0], -1) @ W4.T + b4) @ W5.T + b5


def exact(case, seed):
    kind, L = case["kind"], case.get("L")
    if kind == "energy":
        return _exact_energy(case, seed)
    if kind == "deltas":
        return _exact_deltas(case, seed)
    if kind == "operators":
        return _exact_operators(case, seed)
    if kind == "forward":
        words, flat = _random_words(L, case["n"], seed), _network(L, seed).to(torch.float64)
        with torch.no_grad():
            return torch.cat([_logits(words[i:i + 256], L, flat) for i in range(0, words.shape[0], 256)])
    if kind == "train":
        words, target, weight, lo, hi = _train_batch(case, seed)
        flat = _network(L, seed).to(torch.float64).requires_grad_(True)
        weight = weight.to(torch.float64)
        loss = 0.0
        for i in range(0, words.shape[0], 64):
            free = _logits(words[i:i + 64], L, flat)[:, lo:hi + 1]
            ce = torch.logsumexp(free, 1) - free.gather(1, target[i:i + 64, None].long() - lo)[:, 0]
            part = (weight[i:i + 64] * ce).sum() / weight.sum()
            part.backward()
            loss = loss + part.detach()
        return loss.reshape(1), flat.grad
    return None  # searches: a plain replay of millions of flips or expansions takes far longer than 20 s
