"""The work that a user of this decoder has it do, as measurable cases.

Each case goes through the package's public calls on inputs sampled from its
own noise model: single shots and batches of untruncated decoding, one graph
launch over mixed distances, the truncated sweep at large distance, training
steps through the adjoint, the detector picture, and decoding under independent
X/Z noise. Rates, distances, bond dimensions and batch sizes are those of the
repository's bench and tests, or generic odd sizes next to them.

What comes back is what a program keeps. The sweeps compute in FP32 (ln Z is
only stored in FP64), so ln Z_l of every class is kept in 32 bits. Where classes
far below the leading one are rounding noise of the leading one (truncated
bonds, and determinants of signed terms), a program keeps the posterior
Pr(l|s) and the evidence ln Pr(s) instead, in the precision of the path.
"""
import math

import numpy as np
import torch

import paper_2605_17230_gb300 as mld

DEV = "cuda"


def listed():
    return [
        # one round of a real-time loop on a small patch: pure latency
        {"name": "one shot d=5", "kind": "decode", "d": 5, "chi": 16, "B": 1, "noise": "table", "mixed": False},
        # a rate scan: every shot with its own depolarizing strength, no decisions kept
        {"name": "rate scan d=7", "kind": "decode", "d": 7, "chi": 16, "B": 262_143, "noise": "shots", "mixed": False},
        # the bench's workload: d=9, chi=32, p=0.10, all four classes, mixed precision asked for
        {"name": "headline d=9", "kind": "decode", "d": 9, "chi": 32, "B": 65_536, "noise": "depol", "mixed": True},
        # the largest distance decoded without truncation, a ragged batch
        {"name": "untruncated d=13", "kind": "decode", "d": 13, "chi": 64, "B": 4_099, "noise": "table",
         "mixed": False},
        # a serving batch over all untruncated distances as one graph launch
        {"name": "mixed batch d=3..13", "kind": "graph", "B": 131_072, "mixed": True},
        # large patches below threshold, where the boundary state has to be truncated
        {"name": "truncated d=17", "kind": "trunc", "d": 17, "chi": 32, "B": 2_048, "noise": "depol", "p": 0.12},
        {"name": "truncated d=25", "kind": "trunc", "d": 25, "chi": 64, "B": 515, "noise": "depol", "p": 0.12},
        # fitting a per-qubit noise model to labelled shots (forward and adjoint)
        {"name": "labelled step d=7", "kind": "train", "d": 7, "chi": 32, "B": 65_536, "labels": True},
        # the same from unlabelled shots, at the distance where the adjoint fills an SM
        {"name": "unlabelled step d=11", "kind": "train", "d": 11, "chi": 32, "B": 2_049, "labels": False},
        # a detector error model with X, Y and Z mechanisms on every qubit
        {"name": "detector picture d=9", "kind": "dem", "d": 9, "B": 65_536},
        # independent X/Z noise near threshold, in 32 bits
        {"name": "independent XZ d=17", "kind": "xz", "d": 17, "B": 8_191, "p": 0.10, "fp64": False, "bitflip": False},
        # the same noise at a lower rate on the largest patch, where 64 bits are asked for
        {"name": "independent XZ d=25", "kind": "xz", "d": 25, "B": 700, "p": 0.05, "fp64": True, "bitflip": False},
    ]


def _log_uniform(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["decode", "decode", "decode", "graph", "trunc", "trunc", "train", "train", "dem", "xz", "xz"])
    if kind == "decode":
        d = rng.choice([3, 5, 7, 9, 11, 13])
        most = {3: 1_000_000, 5: 1_000_000, 7: 1_000_000, 9: 400_000, 11: 100_000, 13: 20_000}[d]
        return {"kind": kind, "d": d, "chi": rng.choice([c for c in (16, 32, 64) if c >= 2 ** (d // 2)]),
                "B": _log_uniform(rng, 1, most), "noise": rng.choice(["table", "shots"]), "mixed": rng.random() < 0.4}
    if kind == "graph":
        return {"kind": kind, "B": _log_uniform(rng, 600, 120_000), "mixed": rng.random() < 0.5}
    if kind == "trunc":
        d = rng.choice([9, 11, 13, 17, 21, 25])
        chi = {9: [8], 11: [8, 16], 13: [16, 32], 17: [16, 32, 64, 128], 21: [32, 64], 25: [32, 64, 128]}[d]
        most = {9: 8_000, 11: 3_000, 13: 2_500, 17: 1_800, 21: 800, 25: 400}[d]
        return {"kind": kind, "d": d, "chi": rng.choice(chi), "B": _log_uniform(rng, 1, most),
                "noise": rng.choice(["depol", "biased"]), "p": round(rng.uniform(0.04, 0.12), 3)}
    if kind == "train":
        d = rng.choice([3, 5, 7, 9, 11, 13])
        most = {3: 200_000, 5: 120_000, 7: 65_000, 9: 30_000, 11: 8_000, 13: 800}[d]
        return {"kind": kind, "d": d, "chi": max(32, 2 ** (d // 2)), "B": _log_uniform(rng, 16, most),
                "labels": rng.random() < 0.5}
    if kind == "dem":
        d = rng.choice([3, 5, 7, 9, 11])
        most = {3: 500_000, 5: 500_000, 7: 300_000, 9: 65_000, 11: 20_000}[d]
        return {"kind": kind, "d": d, "B": _log_uniform(rng, 1, most)}
    # FP32 is the near-threshold mode; 64 bits at any rate
    fp64 = rng.random() < 0.4
    d = rng.choice([5, 9, 13, 17, 21, 25] if fp64 else [5, 9, 11, 13, 15, 17])
    most = {5: 40_000, 9: 20_000, 11: 12_000, 13: 8_000, 15: 6_000, 17: 8_000, 21: 1_000, 25: 500}[d]
    return {"kind": "xz", "d": d, "B": _log_uniform(rng, 1, most // (8 if fp64 and d < 21 else 1)),
            "p": round(rng.uniform(0.02, 0.12) if fp64 else rng.uniform(0.09, 0.12), 3), "fp64": fp64,
            "bitflip": rng.random() < 0.3}


# ---------------------------------------------------------------- inputs ---

def _checks(d):
    """Check matrices of the rotated patch, in the library's documented order:
    bits of a row are the qubits whose z (X-type) or x (Z-type) part it sees."""
    rows = []
    for j in range(d + 1):
        for i in range(d + 1):
            xtype = (i + j) % 2 == 0
            inside = 1 <= i < d and 1 <= j < d
            edge = (i in (0, d) and 1 <= j < d and xtype) or (j in (0, d) and 1 <= i < d and not xtype)
            if inside or edge:
                rows.append((xtype, [r * d + c for r in (i - 1, i) for c in (j - 1, j) if 0 <= r < d and 0 <= c < d]))
    hx = np.zeros((len(rows), d * d), np.float32)        # sees x parts
    hz = np.zeros_like(hx)
    for k, (xtype, qs) in enumerate(rows):
        (hz if xtype else hx)[k, qs] = 1
    return torch.from_numpy(hx).to(DEV), torch.from_numpy(hz).to(DEV)


def _syndromes(d, x, z):
    hx, hz = _checks(d)
    bits = (x.float() @ hx.T + z.float() @ hz.T).to(torch.int64) & 1
    words = (bits.shape[1] + 63) // 64
    out = torch.zeros((x.shape[0], words), dtype=torch.int64, device=DEV)
    for w in range(words):
        part = bits[:, 64 * w:64 * w + 64]
        out[:, w] = (part << torch.arange(part.shape[1], device=DEV)).sum(1)
    return out


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _lognormal_table(n, g):
    """Calibrated per-qubit rates: median 0.05, sigma 0.5, Z bias 1..10."""
    p = (0.05 * torch.exp(0.5 * torch.randn(n, generator=g, device=DEV, dtype=torch.float64))).clamp(1e-4, 0.45)
    eta = 1 + 9 * torch.rand(n, generator=g, device=DEV, dtype=torch.float64)
    side = p / (2 * (1 + eta))
    return torch.stack([1 - p, side, side, p * eta / (1 + eta)], 1)


def _sample(table, B, g):
    """x and z bits [B][n] of errors from a table [n][4] of rows (I, X, Y, Z)."""
    cum = torch.cumsum(table.float(), -1)
    u = torch.rand((B, table.shape[0]), generator=g, device=DEV)
    x = (u >= cum[..., 0]) & (u < cum[..., 2])
    z = (u >= cum[..., 1]) & (u < 1.0)
    return x, z


def _shots(d, B, g):
    """Depolarizing strengths in [0.02, 0.18], one per shot, and their errors."""
    p = 0.02 + 0.16 * torch.rand(B, generator=g, device=DEV)
    u = torch.rand((B, d * d), generator=g, device=DEV)
    q = p[:, None]
    return p, (u < 2 * q / 3), (u >= q / 3) & (u < q)


def _depol(n, p):
    return torch.tensor([[1 - p, p / 3, p / 3, p / 3]], dtype=torch.float64, device=DEV).repeat(n, 1)


def _biased(n, p, eta):
    side = p / (2 * (1 + eta))
    return torch.tensor([[1 - p, side, side, p * eta / (1 + eta)]], dtype=torch.float64, device=DEV).repeat(n, 1)


def _table_of(case, n, g):
    if case.get("noise") == "depol":
        return _depol(n, case.get("p", 0.10))
    if case.get("noise") == "biased":
        return _biased(n, case["p"], 100.0)
    return _lognormal_table(n, g)


def _xz_rates(case, n, g):
    px = case["p"] * (0.8 + 0.4 * torch.rand(n, generator=g, device=DEV))
    pz = case["p"] * (0.8 + 0.4 * torch.rand(n, generator=g, device=DEV))
    return px, None if case["bitflip"] else pz


def _mechanisms(n, g):
    q = torch.arange(n).repeat_interleave(3).numpy().astype(np.int32)
    c = np.tile(np.array([1, 2, 3], np.int32), n)
    p = (0.03 * torch.exp(0.5 * torch.randn(3 * n, generator=g, device=DEV, dtype=torch.float64))).clamp(1e-4, 0.3)
    return q, c, p


def _inputs(case, seed):
    """Noise, error bits and syndromes of a case, all from the seed."""
    g = _gen(seed)
    d, B = case["d"], case["B"]
    n = d * d
    kind = case["kind"]
    if kind == "dem":
        q, c, p = _mechanisms(n, g)
        x = torch.zeros((B, n), dtype=torch.bool, device=DEV)
        z = torch.zeros_like(x)
        for k, pauli in enumerate((1, 2, 3)):
            hit = torch.rand((B, n), generator=g, device=DEV) < p[k::3].float()
            x ^= hit & bool(pauli & 1)
            z ^= hit & bool(pauli & 2)
        noise = (q, c, p)
    elif kind == "xz":
        px, pz = _xz_rates(case, n, g)
        x = torch.rand((B, n), generator=g, device=DEV) < px
        z = torch.rand((B, n), generator=g, device=DEV) < (0.0 if pz is None else pz)
        noise = (px, pz)
    elif case.get("noise") == "shots":
        noise, x, z = _shots(d, B, g)
    else:
        noise = _table_of(case, n, g).float()
        x, z = _sample(noise, B, g)
    return noise, x, z, _syndromes(d, x, z)


GRAPH_CHI = {3: 16, 5: 16, 7: 16, 9: 32, 11: 32, 13: 64}


def _graph_jobs(case):
    """One job per distance; a sixth of the batch each, the last ones ragged."""
    share = max(1, case["B"] // 6)
    return [{"kind": "decode", "d": d, "chi": chi, "B": max(1, share - 7 * k), "noise": "table",
             "mixed": case["mixed"]} for k, (d, chi) in enumerate(GRAPH_CHI.items())]


def _precision(case):
    return mld.MLD_MIXED_TF32 if case["mixed"] else mld.MLD_FP32


def prepare(case, seed):
    if case["kind"] == "graph":
        items = []
        for k, job in enumerate(_graph_jobs(case)):
            noise, _, _, syn = _inputs(job, seed * 8 + k)
            lp = torch.empty((job["B"], 4), dtype=torch.float64, device=DEV)
            am = torch.empty((job["B"],), dtype=torch.uint8, device=DEV)
            items.append((mld.Code(job["d"]), noise, syn, job["chi"], _precision(case), lp, am))
        return {"case": case, "items": items, "graph": mld.Graph(mld.make_jobs(items))}
    noise, x, z, syn = _inputs(case, seed)
    state = {"case": case, "code": mld.Code(case["d"]), "noise": noise, "syn": syn}
    if case["kind"] == "dem":
        state["noise"] = (noise[0], noise[1], noise[2].cpu().numpy())
    if case["kind"] == "train":
        state["noise"] = noise.requires_grad_(True)
        state["true"] = _class_of(case["d"], x, z)[:, None]
    return state


def _class_of(d, x, z):
    lx = x[:, :d].sum(1) & 1                              # x parity on row 0
    lz = z[:, ::d].sum(1) & 1                             # z parity on column 0
    return lx + 2 * lz


# ------------------------------------------------------------------- run ---

def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "graph":
        state["graph"].launch()
        return [(it[5].float(), it[6]) for it in state["items"]]
    code, noise, syn = state["code"], state["noise"], state["syn"]
    if kind == "decode":
        # no decisions are kept of shots with one rate each: uniform noise ties exactly on small patches
        lp, am = code.decode(noise, syn, case["chi"], _precision(case), with_argmax=case["noise"] != "shots")
        return (lp.float(),) if am is None else (lp.float(), am)
    if kind == "trunc":
        lp, am = code.decode(noise, syn, case["chi"])
        return torch.softmax(lp, 1).float(), torch.logsumexp(lp, 1).float(), am
    if kind == "dem":
        lp, am = code.decode_dem(*noise, syn)
        return lp.float(), am
    if kind == "xz":
        lp, am = code.decode_xz(*noise, syn, mld.MLD_FP64 if case["fp64"] else mld.MLD_FP32)
        post, evidence = torch.softmax(lp, 1), torch.logsumexp(lp, 1)
        return (post, evidence, am) if case["fp64"] else (post.float(), evidence.float(), am)
    noise.grad = None
    lp = mld.log_coset_probabilities(code, noise, syn, case["chi"])
    _loss(lp, state["true"] if case["labels"] else None).backward()
    return noise.grad, lp.detach().float()


def _loss(lp, true):
    """-mean ln Pr(true class | s) of labelled shots, or -mean ln Pr(s)."""
    evidence = torch.logsumexp(lp, 1)
    return -evidence.mean() if true is None else (evidence - lp.gather(1, true)[:, 0]).mean()


# ------------------------------------------------------------------ work ---

def work(case):
    """Inputs read once and outputs written once; the flops of the exact column
    transfer (two classes share all columns but the last; three flops an entry
    and qubit), of a backward pass twice that again, and for a truncated sweep
    those of bonds of six."""
    if case["kind"] == "graph":
        parts = [work(j) for j in _graph_jobs(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    d, B, kind = case["d"], case["B"], case["kind"]
    n = d * d
    nbytes = B * (8 * ((n - 1 + 63) // 64) + 32 + 1) + 16 * n
    if case.get("noise") == "shots":
        nbytes += 4 * B - 16 * n
    columns = 2 * (n - d) + 4 * d
    if kind == "trunc":
        return {"bytes": nbytes, "flops": B * columns * 40.0 * 6 ** 3}
    if kind == "xz":
        return {"bytes": nbytes, "flops": B * (1 if case["bitflip"] else 2) * (n + d) * 3.0 * 2 ** ((d - 1) // 2)}
    flops = B * columns * 3.0 * 2 ** d
    if kind == "train":
        return {"bytes": nbytes + 32 * B + 32 * n, "flops": 3 * flops}
    return {"bytes": nbytes, "flops": flops}


# ----------------------------------------------------------------- exact ---

def _transfer(d, w):
    """ln Z [U] by the exact column transfer in FP64: w[U][n][x][z] holds the
    probability of the Pauli that x, z and the representative give. One bit per
    row position: in an even column position r turns from the check above-left
    of qubit (r, c) into the one below-right of it, rows in rising order; in an
    odd one from below-left to above-right, in falling order. Position r is
    X-type for even r; its neighbours r-1, r+1 are of the other type."""
    U = w.shape[0]
    even = sum(1 << k for k in range(0, d, 2))
    idx = torch.arange(1 << d, device=w.device)
    ends = ((idx & even) == 0).to(w.dtype)               # no X-type check on the first and last corner column
    S = ends[None].expand(U, -1)
    lnz = torch.zeros(U, dtype=w.dtype, device=w.device)
    for c in range(d):
        for r in range(d) if c % 2 == 0 else range(d - 1, -1, -1):
            q = w[:, r * d + c]                          # [U][x][z]
            q = q if r % 2 == 0 else q.transpose(1, 2)   # [U][flip][control]
            up, down = (2 if r + 1 < d else 1), (2 if r > 0 else 1)
            S = S.reshape(U, -1, up, 2, down, (1 << r) // down)
            a = torch.arange(up, device=w.device)[:, None] ^ torch.arange(down, device=w.device)[None]
            k = q[:, :, a]                               # [U][flip][up][down]
            same, flip = (k[:, f][:, None, :, None, :, None] for f in (0, 1))
            S = same * S + flip * S.flip(3)
        S = S.reshape(U, -1)
        top = S.detach().amax(1, keepdim=True)
        S = S / top
        lnz = lnz + torch.log(top[:, 0])
    return lnz + torch.log((S * ends).sum(1))


def _class_weights(d, table, x, z):
    """w[B*4][n][x][z] of the four classes, from errors x, z as representatives
    (class l is reached from the error's own class by X on column 0 and Z on
    row 0). table: [n][4] or [B][n][4] rows (I, X, Y, Z)."""
    B, n = x.shape
    own = _class_of(d, x, z)
    l = torch.arange(4, device=x.device)[None] ^ own[:, None]                     # [B][4]
    col0 = torch.zeros(n, dtype=torch.bool, device=x.device)
    row0 = col0.clone()
    col0[::d], row0[:d] = True, True
    ex = x[:, None] ^ ((l & 1).bool()[..., None] & col0)
    ez = z[:, None] ^ ((l & 2).bool()[..., None] & row0)
    pauli = torch.tensor([[0, 3], [1, 2]], device=x.device)                        # [x][z] -> I, Z / X, Y
    e = torch.arange(2, device=x.device)
    at = pauli[ex.long()[..., None, None] ^ e[:, None], ez.long()[..., None, None] ^ e[None]]   # [B][4][n][2][2]
    rows = table.expand(B, n, 4)[:, None].expand(B, 4, n, 4)
    return torch.gather(rows, 3, at.reshape(B, 4, n, 4)).reshape(B * 4, n, 2, 2)


def _chunks(B, each):
    return [(b, min(B, b + each)) for b in range(0, B, each)]


def _exact_lnz(d, table, x, z):
    """ln Z [B][4] in FP64, chunk by chunk."""
    out = torch.empty((x.shape[0], 4), dtype=torch.float64, device=x.device)
    for a, b in _chunks(x.shape[0], max(1, (1 << 27) >> d)):
        t = table if table.dim() == 2 else table[a:b]
        out[a:b] = _transfer(d, _class_weights(d, t, x[a:b], z[a:b])).reshape(-1, 4)
    return out


def _part(d, p, e, turned):
    """ln of the X part's two sums [B][2] (the sum over x patterns of one
    syndrome, without and with the logical string, relative to the error e):
    the transfer with only the other type's checks as state is the general one
    with z parts free, so it is run here on half the positions."""
    B, n = e.shape
    grid = torch.arange(n, device=e.device).reshape(d, d)
    # the Z-type checks of a patch are the X-type ones of the patch turned by a quarter
    order = torch.flip(grid, (0,)).T.reshape(-1) if turned else grid.reshape(-1)
    p, e = p[order].double(), e[:, order]
    string = torch.zeros(n, dtype=torch.bool, device=e.device)
    string[d - 1::d] = True                              # the last column
    e2 = torch.stack([e, e ^ string], 1).reshape(2 * B, n)
    w = torch.stack([torch.where(e2, p, 1 - p), torch.where(e2, 1 - p, p)], 2)     # [U][n][check parity]
    U, h = 2 * B, (d + 1) // 2                           # positions 0, 2, .., d-1 of the general transfer
    first = (torch.arange(1 << h, device=e.device) == 0).double()
    S = first[None].expand(U, -1)
    lnz = torch.zeros(U, dtype=torch.float64, device=e.device)
    for c in range(d):
        for r in range(d) if c % 2 == 0 else range(d - 1, -1, -1):
            q = w[:, r * d + c]
            k = r // 2
            if r % 2 == 0:
                S = S.reshape(U, -1, 2, 1 << k)
                S = q[:, 0, None, None, None] * S + q[:, 1, None, None, None] * S.flip(2)
            else:
                S = S.reshape(U, -1, 2, 2, 1 << k)       # bits k+1 and k
                a = torch.arange(2, device=e.device)
                S = S * q[:, a[:, None] ^ a[None]][:, None, :, :, None]
        S = S.reshape(U, -1)
        top = S.amax(1, keepdim=True)
        S = S / top
        lnz = lnz + torch.log(top[:, 0])
    return (lnz + torch.log(S[:, 0])).reshape(B, 2)


def _exact_xz(case, noise, x, z):
    d, (px, pz) = case["d"], noise
    own = _class_of(d, x, z)
    zx = torch.cat([_part(d, px, x[a:b], False) for a, b in _chunks(x.shape[0], 2048)])
    if pz is None:                                       # the class of the identity on z parts alone
        zz = torch.stack([torch.zeros_like(zx[:, 0]), torch.full_like(zx[:, 0], -math.inf)], 1)
    else:
        zz = torch.cat([_part(d, pz, z[a:b], True) for a, b in _chunks(x.shape[0], 2048)])
    l = torch.arange(4, device=x.device)[None] ^ own[:, None]
    return zx.gather(1, l & 1) + zz.gather(1, l >> 1)


def exact(case, seed):
    kind = case["kind"]
    if kind == "graph":
        out = []
        for k, job in enumerate(_graph_jobs(case)):
            noise, x, z, _ = _inputs(job, seed * 8 + k)
            out.append((_exact_lnz(job["d"], noise.double(), x, z), None))
        return out
    d, B = case["d"], case["B"]
    if kind == "trunc" and (d > 17 or (B << d) > (1 << 28)):
        return None                                      # the untruncated state is too large for seconds
    noise, x, z, _ = _inputs(case, seed)
    if kind == "xz":
        lp = _exact_xz(case, noise, x, z)
    elif kind == "dem":
        t = torch.zeros((d * d, 4), dtype=torch.float64, device=DEV)
        t[:, 0] = 1
        for k, swap in enumerate(([1, 0, 3, 2], [3, 2, 1, 0], [2, 3, 0, 1])):      # X, Z, Y on (I, X, Y, Z)
            p = noise[2][k::3, None]
            t = (1 - p) * t + p * t[:, swap]
        lp = _exact_lnz(d, t, x, z)
    elif kind == "train":
        return _exact_step(case, noise, x, z)
    elif case["noise"] == "shots":
        p = noise.double()[:, None, None]
        t = torch.cat([1 - p, p / 3, p / 3, p / 3], 2).expand(B, d * d, 4)
        lp = _exact_lnz(d, t, x, z)
    else:
        lp = _exact_lnz(d, noise.double(), x, z)
    if kind in ("trunc", "xz"):
        return torch.softmax(lp, 1), torch.logsumexp(lp, 1), None
    return (lp,) if kind == "decode" and case["noise"] == "shots" else (lp, None)


def _exact_step(case, noise, x, z):
    """Gradient and ln Z of a training step by FP64 automatic differentiation,
    as many shots at a time as the saved states leave room for."""
    d, B = case["d"], case["B"]
    table = noise.detach().double().requires_grad_(True)
    true = _class_of(d, x, z)[:, None]
    out = torch.empty((B, 4), dtype=torch.float64, device=x.device)
    each = max(1, int(24e9 / (4 * d * d * 32.0 * 2 ** d)))
    for a, b in _chunks(B, each):
        lp = _transfer(d, _class_weights(d, table, x[a:b], z[a:b])).reshape(-1, 4)
        (_loss(lp, true[a:b] if case["labels"] else None) * ((b - a) / B)).backward()
        out[a:b] = lp.detach()
    return table.grad, out
