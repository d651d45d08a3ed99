"""The calls whose speed is followed: what a program that validates Gaussian
boson sampling data has this library do, over the range of its sizes.

A case is a dict of plain values with a "kind":
  counts     gbs_reset + gbs_sample + gbs_binned_counts on a resident network
             (with fresh=True: gbs_make_network from page-locked host memory,
             the same two calls, gbs_free_network)
  moments    gbs_moments: normally-ordered moments and single-mode marginals
  binned     gbs_sample_nd + gbs_binned_counts_nd: joint count distribution of
             d output bins
  batch      gbs_sample_batch + gbs_binned_counts over uneven networks
  predict    Surrogate.predict: distributions of many networks from the MLP
  train      gbs_mlp_train: Adam steps on a training set
listed() are the ones looked at one by one, draw() gives others of the same
ranges.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2503_12749_gb300 as gbs
from paper_2503_12749_gb300 import surrogate

DEV = "cuda"


def listed():
    return [
        # Smallest: the plain FP64 run that is checked against the closed form.
        dict(name="small16_fp64", kind="counts", precision="fp64", N=16, M=16, r_lo=1.0, r_hi=1.0,
             t2=0.9, E=2**14, n_sub=16, K1=64, m_offset=0, fresh=False),
        # FP64 reference run of the 1000-mode low-loss network, against which the
        # split-precision runs are judged.
        dict(name="m1000_fp64", kind="counts", precision="fp64", N=1000, M=1000, r_lo=1.0, r_hi=1.0,
             t2=0.98, E=2**15, n_sub=100, K1=4096, m_offset=0, fresh=False),
        # FP32 run of a rectangular network of no round size (part of the modes detected).
        dict(name="ragged_fp32", kind="counts", precision="fp32", N=700, M=615, r_lo=0.5, r_hi=1.0,
             t2=0.95, E=20001, n_sub=37, K1=2048, m_offset=0, fresh=False),
        # Production run of the 1000-mode network: 10^6 trajectories, sub-ensembles of 10^4.
        dict(name="m1000_bf16x3", kind="counts", precision="bf16x3", N=1000, M=1000, r_lo=1.0,
             r_hi=1.0, t2=0.98, E=10**6, n_sub=100, K1=4096, m_offset=0, fresh=False),
        # A new network each time, odd sizes, non-uniform squeezing: the whole
        # program from T in host memory to P(m) in host memory.
        dict(name="fresh_ragged_bf16x3", kind="counts", precision="bf16x3", N=333, M=517, r_lo=0.5,
             r_hi=1.5, t2=0.9, E=100003, n_sub=64, K1=2048, m_offset=0, fresh=True),
        # The largest single-GPU network, part of its 2^20 trajectories.
        dict(name="m8000_bf16x3", kind="counts", precision="bf16x3", N=8000, M=8000, r_lo=1.0,
             r_hi=1.0, t2=0.99, E=2**17, n_sub=64, K1=16384, m_offset=2754, fresh=False),
        # The six-product accuracy mode.
        dict(name="m1000_bf16x6", kind="counts", precision="bf16x6", N=1000, M=1000, r_lo=1.0,
             r_hi=1.0, t2=0.98, E=2**17, n_sub=64, K1=4096, m_offset=0, fresh=False),
        # Per-mode moments and marginals of every output mode.
        dict(name="moments_m1000_bf16x3", kind="moments", precision="bf16x3", N=1000, M=1000,
             r_lo=1.0, r_hi=1.0, t2=0.98, E=2**18, n_sub=100, mmax=4, cmax=7),
        # The two-bin example of the paper (Fig. 3): lossless, 200 modes, 1.2e6 samples.
        dict(name="bin2d_200_bf16x3", kind="binned", precision="bf16x3", N=200, M=200, r_lo=0.5,
             r_hi=0.5, t2=1.0, bins=2, E=1200000, n_sub=100, K=128),
        # Many networks of uneven size in one call.
        dict(name="batch16_bf16x3", kind="batch", precision="bf16x3", count=16, n_lo=100, n_hi=2000,
             E=2**16, n_sub=64, sizes=1),
        # Surrogate prediction of 51 networks (50 held-out ones and the largest).
        dict(name="predict51", kind="predict", count=51, n_lo=500, n_hi=8000, sizes=2),
        # Surrogate training: one of 40 rounds of the 400 Adam steps, 1800 networks.
        dict(name="train1800", kind="train", rows=1800, steps=10),
    ]


def draw(rng):
    kind = rng.choices(["counts", "moments", "binned", "batch", "predict", "train"],
                       [10, 2, 2, 1, 1, 1])[0]

    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    if kind == "predict":
        return dict(kind=kind, count=log(1, 500), n_lo=500, n_hi=rng.choice([2000, 8000]),
                    sizes=rng.randrange(1000))
    if kind == "train":
        return dict(kind=kind, rows=log(100, 2000), steps=rng.randint(5, 15))
    if kind == "batch":
        return dict(kind=kind, precision=rng.choice(["bf16x3", "bf16x3", "bf16x6"]),
                    count=rng.randint(2, 16), n_lo=100, n_hi=log(300, 2000), E=log(2**13, 2**16),
                    n_sub=rng.randint(10, 64), sizes=rng.randrange(1000))
    if kind == "binned":
        precision = rng.choice(["bf16x3", "bf16x3", "fp64"])
        bins = rng.choice([2, 2, 3])
        return dict(kind=kind, precision=precision, N=log(8, 200), M=log(8, 200), r_lo=0.3,
                    r_hi=round(rng.uniform(0.3, 0.6), 3), t2=rng.choice([1.0, 0.95]), bins=bins,
                    E=log(2000, 20000 if precision == "fp64" else 1200000 if bins == 2 else 50000),
                    n_sub=rng.randint(10, 100), K=128 if bins == 2 else 32)
    precision = rng.choice(["fp64", "fp64", "fp32", "bf16x3", "bf16x3", "bf16x3", "bf16x6"])
    simt = precision in ("fp64", "fp32")
    N = log(16, 1500 if simt or kind == "moments" else 8000)
    M = N if rng.random() < 0.5 else max(8, int(N * rng.uniform(0.5, 1.5)))
    flop = 2.6e11 if precision == "fp64" else 5e11 if precision == "fp32" else 2e13
    E = max(1000, min(log(2**12, 10**6 if not simt else 2**17), int(flop / (8.0 * M * N))))
    r_lo = round(rng.uniform(0.5, 1.2), 3)
    r_hi = r_lo if rng.random() < 0.5 else round(r_lo + rng.uniform(0.0, 0.4), 3)
    t2 = round(rng.uniform(0.25, 0.99), 3)
    n_sub = rng.randint(10, 128)
    if kind == "moments":
        if precision == "fp64":
            E = min(E, 2**15)
        return dict(kind=kind, precision=precision, N=N, M=M, r_lo=r_lo, r_hi=r_hi, t2=t2,
                    E=min(E, 2**18), n_sub=n_sub, mmax=rng.randint(1, 6), cmax=rng.randint(1, 9))
    K1, m_offset = count_window(r_lo, r_hi, N, t2 * min(1.0, M / N))
    return dict(kind=kind, precision=precision, N=N, M=M, r_lo=r_lo, r_hi=r_hi, t2=t2, E=E,
                n_sub=n_sub, K1=K1, m_offset=m_offset, fresh=rng.random() < 0.3 and M * N <= 4000000)


def count_window(r_lo, r_hi, N, t2):
    """(K1, m_offset): 12 standard deviations of the total count about its mean."""
    s2 = math.sinh(0.5 * (r_lo + r_hi)) ** 2
    c2 = math.cosh(r_hi) ** 2
    half = 12.0 * math.sqrt(N * (t2 * (1.0 - t2) * s2 + 2.0 * t2 * t2 * math.sinh(r_hi) ** 2 * c2)) + 64
    K1 = 1 << int(math.ceil(math.log2(2.0 * half)))
    return K1, max(0, int(t2 * N * s2) - K1 // 2)


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def unitary(n, gen):
    """A random n x n unitary on the GPU: Haar (QR) up to 1024 modes, above it
    the product F D2 F D1 of Fourier matrices and random phases."""
    if n <= 1024:
        z = torch.randn(n, n, 2, generator=gen, dtype=torch.float64, device=DEV)
        q, r = torch.linalg.qr(torch.view_as_complex(z))
        d = torch.diagonal(r)
        return q * (d / d.abs())[None, :]
    ph = torch.rand(2, n, generator=gen, dtype=torch.float64, device=DEV) * (2.0 * math.pi)
    d = torch.polar(torch.ones_like(ph), ph)
    u = torch.fft.fft(torch.diag(d[0]), dim=0, norm="ortho")
    return torch.fft.fft(d[1][:, None] * u, dim=0, norm="ortho")


def generator(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def network(c, seed, N, M):
    """(T on the GPU, r on the host): M x N part of a unitary with uniform loss."""
    U = unitary(max(N, M), generator(seed))[:M, :N]
    rng = np.random.default_rng(seed)
    r = rng.uniform(c["r_lo"], c["r_hi"], size=N) if c["r_hi"] > c["r_lo"] else np.full(N, c["r_lo"])
    return (math.sqrt(c["t2"]) * U).contiguous(), r


def batch_parts(c, seed):
    """Per network of the batch: (case of its counts, seed)."""
    rng = np.random.default_rng(c["sizes"])
    out = []
    for i in range(c["count"]):
        n = int(round(math.exp(rng.uniform(math.log(c["n_lo"]), math.log(c["n_hi"])))))
        t = float(rng.uniform(0.5, 0.995))
        K1, m_off = count_window(0.5, 1.5, n, t * t)
        out.append((dict(precision=c["precision"], N=n, M=n, r_lo=0.5, r_hi=1.5, t2=t * t, E=c["E"],
                         n_sub=c["n_sub"], K1=K1, m_offset=m_off), 1000 * seed + i))
    return out


class SurrogateNet:
    """What Surrogate.predict reads of a network: size, loss and range of the
    squeezing from `sizes`, the squeezing itself from `rng`."""

    def __init__(self, sizes, rng, n_lo, n_hi):
        self.N = self.M = int(round(math.exp(sizes.uniform(math.log(n_lo), math.log(n_hi)))))
        mid, dev = sizes.uniform(0.5, 1.5), sizes.uniform(0.0, 0.3)
        self.t = float(sizes.uniform(0.9, 0.999))
        self.r = rng.uniform(mid - dev, mid + dev, size=self.N)
        self.K1, self.m_off = count_window(mid - dev, mid + dev, self.N, self.t**2)


def surrogate_nets(c, seed):
    """(100 networks that set the feature statistics, the case's networks)."""
    sizes, rng = np.random.default_rng(c["sizes"]), np.random.default_rng(seed)
    nets = [SurrogateNet(sizes, rng, c["n_lo"], c["n_hi"]) for _ in range(100 + c["count"])]
    return nets[:100], nets[100:]


def mlp_weights(seed):
    """He-normal weights of the 10-512-512-512-512 MLP, rounded to BF16, packed."""
    rng = np.random.default_rng(seed)
    dims, parts = [10, 512, 512, 512, 512], []
    for i in range(4):
        W = rng.normal(size=(dims[i + 1], dims[i])) * math.sqrt(2.0 / dims[i]) * (0.1 if i == 3 else 1.0)
        parts += [W.ravel(), 0.1 * rng.normal(size=dims[i + 1])]
    return torch.from_numpy(np.concatenate(parts)).to(torch.bfloat16).float().numpy()


def training_set(c, seed):
    """(X, targets, parameters, learning rates): standardised features and the
    density residuals of skewed normal distributions with sampling noise."""
    rng = np.random.default_rng(seed)
    X = rng.normal(size=(c["rows"], 10))
    x = -8.0 + 16.0 * (np.arange(256) + 0.5) / 256
    half_phi = 0.5 * np.exp(-0.5 * x * x) / math.sqrt(2.0 * math.pi)
    skew = 0.1 + 0.05 * X[:, :1] - 0.03 * X[:, 1:2] * X[:, 2:3]
    Y = 100.0 * np.tile(skew * (x**3 - 3 * x) / 6 * half_phi, (1, 2))
    Y += 0.02 * rng.normal(size=Y.shape)
    lr = np.linspace(1e-3, 8e-4, c["steps"]).astype(np.float32)
    return X.astype(np.float32), Y.astype(np.float32), mlp_weights(seed + 1), lr


def prepare(case, seed):
    c = case
    s = dict(case=c, seed=2503 * 10**6 + seed)
    stream = torch.cuda.Stream()
    s["stream"] = stream
    st = stream.cuda_stream
    if c["kind"] == "counts":
        T, r = network(c, seed, c["N"], c["M"])
        if c["fresh"]:
            host = torch.empty(T.shape, dtype=T.dtype, pin_memory=True)
            host.copy_(T)
            s.update(host=host, T=host.numpy(), r=r)
        else:
            torch.cuda.synchronize()
            s["net"] = gbs.gbs_make_network_device(T.data_ptr(), c["M"], c["N"], r, c["precision"], st)
    elif c["kind"] == "moments":
        T, r = network(c, seed, c["N"], c["M"])
        torch.cuda.synchronize()
        s["net"] = gbs.gbs_make_network_device(T.data_ptr(), c["M"], c["N"], r, c["precision"], st)
    elif c["kind"] == "binned":
        T, r = network(c, seed, c["N"], c["M"])
        s["net"] = gbs.gbs_make_network_binned(T.cpu().numpy(), r, bin_of_mode(c), c["precision"], st)
    elif c["kind"] == "batch":
        s["parts"], s["nets"] = [], []
        for part, sd in batch_parts(c, seed):
            T, r = network(part, sd, part["N"], part["M"])
            torch.cuda.synchronize()
            s["nets"].append(gbs.gbs_make_network_device(T.data_ptr(), part["M"], part["N"], r,
                                                         part["precision"], st))
            s["parts"].append(part)
        s["batch"] = gbs.gbs_make_batch(s["nets"])
    elif c["kind"] == "predict":
        known, nets = surrogate_nets(c, seed)
        sur = surrogate.Surrogate(max_batch=2048, stream=stream)
        feat = sur.records(known)
        gbs.gbs_surrogate_feature_stats(len(known), feat.data_ptr(), sur.stats.data_ptr(), st)
        gbs.gbs_mlp_set_params(sur.mlp, mlp_weights(seed))
        sur.trained = True
        s.update(sur=sur, nets=nets)
    else:
        X, Y, params, lr = training_set(c, seed)
        s.update(X=torch.from_numpy(X).to(DEV), Y=torch.from_numpy(Y).to(DEV), params=params, lr=lr)
        s["mlp"] = gbs.gbs_mlp_create(10, 512, 512, 4, 2048, st)
        torch.cuda.synchronize()
    return s


def bin_of_mode(c):
    """Consecutive modes to each bin, as evenly as they go."""
    return (np.arange(c["M"]) * c["bins"] // c["M"]).astype(np.int32)


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------
def run(state):
    c, seed = state["case"], state["seed"]
    kind = c["kind"]
    if kind == "counts":
        if c["fresh"]:
            net = gbs.gbs_make_network(state["T"], state["r"], c["precision"],
                                       state["stream"].cuda_stream)
        else:
            net = state["net"]
            gbs.gbs_reset(net)
        gbs.gbs_sample(net, seed, 0, c["E"], c["n_sub"], c["K1"])
        out = gbs.gbs_binned_counts(net, c["m_offset"], c["K1"])
        if c["fresh"]:
            gbs.gbs_free_network(net)
        return out
    if kind == "moments":
        return gbs.gbs_moments(state["net"], seed, 0, c["E"], c["n_sub"], c["mmax"], c["cmax"])
    if kind == "binned":
        K = [c["K"]] * c["bins"]
        gbs.gbs_reset(state["net"])
        gbs.gbs_sample_nd(state["net"], seed, 0, c["E"], c["n_sub"], K)
        return gbs.gbs_binned_counts_nd(state["net"], K)
    if kind == "batch":
        parts, nets = state["parts"], state["nets"]
        for net in nets:
            gbs.gbs_reset(net)
        gbs.gbs_sample_batch(state["batch"], [seed + i for i in range(len(nets))], [0] * len(nets),
                             [p["E"] for p in parts], [p["n_sub"] for p in parts],
                             [p["K1"] for p in parts])
        return [gbs.gbs_binned_counts(n, p["m_offset"], p["K1"]) for n, p in zip(nets, parts)]
    if kind == "predict":
        P, _, in_domain = state["sur"].predict(state["nets"])
        return P, in_domain
    gbs.gbs_mlp_set_params(state["mlp"], state["params"])
    hist = gbs.gbs_mlp_train(state["mlp"], state["X"].data_ptr(), state["Y"].data_ptr(), c["rows"],
                             state["lr"])
    return hist, gbs.gbs_mlp_get_params(state["mlp"])


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------
def work(case):
    """Bytes: inputs read and outputs written once.  FLOPs: 8 M N per
    trajectory for the propagation (in the result's precision, not the
    products that a split issues), 6 FLOP per weight and row and step for a
    training step's three contractions, 2 for a prediction."""
    c = case
    if c["kind"] in ("counts", "moments", "binned"):
        if c["kind"] == "counts":
            outs = 4 * c["K1"]
        elif c["kind"] == "moments":
            outs = 4 * c["M"] * (c["mmax"] + c["cmax"] + 1)
        else:
            outs = 4 * c["K"] ** c["bins"]
        return dict(bytes=16.0 * c["M"] * c["N"] + 8.0 * c["N"] + 8.0 * outs,
                    flops=8.0 * c["M"] * c["N"] * c["E"])
    if c["kind"] == "batch":
        parts = [work(dict(p, kind="counts")) for p, _ in batch_parts(c, 0)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    weights = 10 * 512 + 3 * 512 * 512
    if c["kind"] == "predict":
        nets = surrogate_nets(c, 0)[1]
        return dict(bytes=2.0 * weights + 8.0 * sum(n.N + n.K1 for n in nets),
                    flops=2.0 * weights * c["count"])
    return dict(bytes=8.0 * (weights + 4 * 512) + 4.0 * c["rows"] * 522,
                flops=6.0 * weights * c["rows"] * c["steps"])


# ---------------------------------------------------------------------------
# The same results in 64 bits from plain torch
# ---------------------------------------------------------------------------
def philox_normals(seed, e0, count, N):
    """Two standard normals [count, N] each: Philox-4x32-10 at counter (e, j),
    53-bit uniforms, Box-Muller."""
    mask = 0xFFFFFFFF
    e = torch.arange(e0, e0 + count, dtype=torch.int64, device=DEV)[:, None].expand(count, N)
    x0, x1 = e & mask, (e >> 32) & mask
    x2 = torch.arange(N, dtype=torch.int64, device=DEV)[None, :].expand(count, N)
    x3 = torch.zeros_like(x0)
    k0, k1 = seed & mask, (seed >> 32) & mask
    for _ in range(10):
        p0, p1 = x0 * 0xD2511F53, x2 * 0xCD9E8D57  # products mod 2^64
        x0, x1, x2, x3 = (((p1 >> 32) & mask) ^ x1 ^ k0, p1 & mask,
                          ((p0 >> 32) & mask) ^ x3 ^ k1, p0 & mask)
        k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
    u1 = (((x0 >> 5) * 67108864 + (x1 >> 6)).double() + 0.5) * 2.0**-53
    u2 = (((x2 >> 5) * 67108864 + (x3 >> 6)).double() + 0.5) * 2.0**-53
    rho = torch.sqrt(-2.0 * torch.log(u1))
    return rho * torch.cos(2.0 * math.pi * u2), rho * torch.sin(2.0 * math.pi * u2)


def trajectories(c, T, r, seed, block):
    """Blocks of (first index, n, alpha', beta')."""
    r = torch.from_numpy(np.asarray(r)).to(DEV)
    cp = torch.sqrt(0.5 * torch.sinh(r) * torch.exp(r))
    cm = torch.sqrt(0.5 * torch.sinh(r) * torch.exp(-r))
    Tr, Ti = T.real.T.contiguous(), T.imag.T.contiguous()
    for e0 in range(0, c["E"], block):
        w1, w2 = philox_normals(seed, e0, min(block, c["E"] - e0), c["N"])
        a, b = cp * w1 + cm * w2, cp * w1 - cm * w2
        yield e0, (a * b).sum(1), torch.complex(a @ Tr, a @ Ti), torch.complex(b @ Tr, -(b @ Ti))


def block_of(c, per):
    """Trajectories per block: about 2^25 elements, whole rounds of sub-ensembles."""
    return max(1, (2**25 // max(per, c["N"], c["M"])) // c["n_sub"]) * c["n_sub"]


def add_by_sub(acc, x):
    """acc[r] += the rows of x whose index is r mod n_sub (x starts at r = 0)."""
    n = acc.shape[0]
    full = x.shape[0] // n
    if full:
        acc += x[: full * n].reshape(full, n, *x.shape[1:]).sum(0)
    if x.shape[0] > full * n:
        acc[: x.shape[0] - full * n] += x[full * n:]


def sub_sizes(E, n_sub):
    i = torch.arange(n_sub, device=DEV)
    return (E // n_sub + (i < E % n_sub)).double()


def mean_and_error(x):
    """Over sub-ensembles (dim 0): mean and error of the mean."""
    return x.mean(0).cpu().numpy(), (x.std(0) / math.sqrt(x.shape[0])).cpu().numpy()


def z_minus_1(K):
    th = 2.0 * math.pi * torch.arange(K, dtype=torch.float64, device=DEV) / K
    return torch.complex(-2.0 * torch.sin(0.5 * th) ** 2, torch.sin(th))


def exact_counts(c, T, r, seed):
    z1 = z_minus_1(c["K1"])
    acc = torch.zeros(2, c["n_sub"], c["K1"], dtype=torch.complex128, device=DEV)
    step = max(1, 2**23 // c["K1"] // c["n_sub"]) * c["n_sub"]
    for _, n, a, b in trajectories(c, T, r, seed, block_of(c, 1)):
        nS = (a * b).sum(1)
        for q in range(0, n.shape[0], step):
            m, L = n[q:q + step, None], nS[q:q + step, None] * z1[None, :]
            lo, hi = torch.clamp(2.0 * m, max=0.0), torch.clamp(2.0 * m, min=0.0)
            g = (torch.exp(L + lo) + torch.exp(-L - hi)) / (1.0 + torch.exp(-2.0 * m.abs()))
            add_by_sub(acc[0], g)
            add_by_sub(acc[1], torch.exp(L))
    acc /= sub_sizes(c["E"], c["n_sub"])[None, :, None]
    P = torch.roll(torch.fft.fft(acc, dim=2).real / c["K1"], -(c["m_offset"] % c["K1"]), dims=2)
    return mean_and_error(P[0]) + mean_and_error(P[1])


def exact_moments(c, T, r, seed):
    ns, M, mm, cm = c["n_sub"], c["M"], c["mmax"], c["cmax"]
    mom = torch.zeros(2, ns, M, mm, dtype=torch.float64, device=DEV)
    marg = torch.zeros(2, ns, M, cm + 1, dtype=torch.float64, device=DEV)
    for _, n, a, b in trajectories(c, T, r, seed, max(1, 2**22 // max(c["N"], M) // ns) * ns):
        x, n = a * b, n[:, None]
        den = 1.0 + torch.exp(-2.0 * n.abs())
        up, dn = torch.exp(n - n.abs() - x) / den, torch.exp(-n - n.abs() + x) / den
        p = torch.ones_like(x)
        plus = torch.exp(-x)
        for k in range(max(mm, cm) + 1):
            if k:
                p = p * x
            if 1 <= k <= mm:
                add_by_sub(mom[0, :, :, k - 1], (p.real * torch.tanh(n)) if k % 2 else p.real)
                add_by_sub(mom[1, :, :, k - 1], p.real)
            if k <= cm:
                f = 1.0 / math.factorial(k)
                add_by_sub(marg[0, :, :, k], (p * (up - dn if k % 2 else up + dn)).real * f)
                add_by_sub(marg[1, :, :, k], (p * plus).real * f)
    size = sub_sizes(c["E"], ns)[None, :, None, None]
    (m0, s0), (m1, s1) = [mean_and_error(x) for x in mom / size]
    (g0, t0), (g1, t1) = [mean_and_error(x) for x in marg / size]
    return np.stack([m0, m1]), np.stack([s0, s1]), np.stack([g0, g1]), np.stack([t0, t1])


def exact_binned(c, T, r, seed):
    K, d, ns = c["K"], c["bins"], c["n_sub"]
    z1 = z_minus_1(K)
    bins = torch.from_numpy(bin_of_mode(c)).to(DEV)
    acc = torch.zeros(2, ns, K ** (d - 1), K, dtype=torch.complex128, device=DEV)
    for _, n, a, b in trajectories(c, T, r, seed, max(1, 2**22 // max(c["N"], c["M"], K ** (d - 1)) // ns) * ns):
        x = a * b
        L = [(x[:, bins == q].sum(1))[:, None] * z1[None, :] for q in range(d)]
        first = L[0]
        for q in range(1, d - 1):
            first = (first[:, :, None] + L[q][:, None, :]).reshape(n.shape[0], -1)
        m = n[:, None]
        lo, hi = torch.clamp(2.0 * m, max=0.0), torch.clamp(2.0 * m, min=0.0)
        inv = 1.0 / (1.0 + torch.exp(-2.0 * m.abs()))

        def outer(u, v):  # sum over each sub-ensemble of u[e, k] v[e, l]
            short = -u.shape[0] % ns
            u, v = (torch.nn.functional.pad(torch.view_as_real(w), (0, 0, 0, 0, 0, short)) for w in (u, v))
            u, v = (torch.view_as_complex(w).reshape(-1, ns, w.shape[1]).permute(1, 2, 0) for w in (u, v))
            return u @ v.transpose(1, 2)

        e1, e2 = torch.exp(first), torch.exp(L[-1])
        acc[1] += outer(e1, e2)
        acc[0] += outer(e1 * (torch.exp(lo) * inv), e2) + outer(torch.exp(-first - hi) * inv, torch.exp(-L[-1]))
    acc /= sub_sizes(c["E"], ns)[None, :, None, None]
    P = torch.fft.fftn(acc.reshape(2, ns, *[K] * d), dim=list(range(2, 2 + d))).real / K**d
    return mean_and_error(P[0]) + mean_and_error(P[1])


def unpack(p):
    dims, out, o = [10, 512, 512, 512, 512], [], 0
    for i in range(4):
        w = p[o:o + dims[i] * dims[i + 1]].reshape(dims[i + 1], dims[i])
        o += w.numel()
        out.append((w, p[o:o + dims[i + 1]]))
        o += dims[i + 1]
    return out


def mlp64(params, X):
    h = X
    for i, (w, b) in enumerate(params):
        h = h @ w.T + b
        if i < 3:
            h = torch.nn.functional.silu(h)
    return h


def exact_train(c, seed):
    X, Y, p, lr = training_set(c, seed)
    X, Y, p = (torch.from_numpy(v).double().to(DEV) for v in (X, Y, p))
    m, v, hist = torch.zeros_like(p), torch.zeros_like(p), []
    for i, rate in enumerate(lr):
        q = p.clone().requires_grad_(True)
        loss = ((mlp64(unpack(q), X) - Y) ** 2).mean()
        (g,) = torch.autograd.grad(loss, q)
        hist.append(float(loss))
        m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
        p = p - float(rate) * (m / (1 - 0.9 ** (i + 1))) / (torch.sqrt(v / (1 - 0.999 ** (i + 1))) + 1e-8)
    return np.array(hist), p.cpu().numpy()


def exact_predict(c, seed):
    def record(n):
        s2 = np.sinh(n.r) ** 2
        mu = n.t**2 * s2.sum()
        sd = math.sqrt((n.t**2 * s2 + n.t**4 * s2 * np.cosh(2 * n.r)).sum())
        return [math.log(n.N), math.log(n.M), n.r.mean(), n.r.std(), n.r.min(), n.r.max(), n.t,
                math.log2(n.K1), math.log(mu), math.log(sd)], mu, sd

    known, nets = surrogate_nets(c, seed)
    known = np.array([record(n)[0] for n in known])
    recs = [record(n) for n in nets]
    X = (np.array([q[0] for q in recs]) - known.mean(0)) / known.std(0)
    W = unpack(torch.from_numpy(mlp_weights(seed)).double())
    out = mlp64(W, torch.from_numpy(X)).numpy().reshape(-1, 2, 256)
    x = -8.0 + 16.0 * (np.arange(256) + 0.5) / 256
    f = out / 100.0 + 0.5 * np.exp(-0.5 * x * x) / math.sqrt(2.0 * math.pi)
    P = np.zeros((len(nets), max(n.K1 for n in nets)))
    for i, (n, (_, mu, sd)) in enumerate(zip(nets, recs)):
        m = n.m_off + np.arange(n.K1)
        g = ((m - mu) / sd - x[0]) * 16.0
        k = np.floor(g).astype(int)
        u = g - k
        y = []
        for d in (-1, 0, 1, 2):
            inside = (k + d >= 0) & (k + d < 256)
            y.append(np.where(inside, f[i][m & 1, np.clip(k + d, 0, 255)], 0.0))
        v = ((2 * u**3 - 3 * u**2 + 1) * y[1] + (u**3 - 2 * u**2 + u) * 0.5 * (y[2] - y[0])
             + (-2 * u**3 + 3 * u**2) * y[2] + (u**3 - u**2) * 0.5 * (y[3] - y[1]))
        v = np.where((g >= 0) & (g <= 255), np.maximum(v, 0.0), 0.0)
        P[i, :n.K1] = v / v.sum()
    return P, None


def exact(case, seed):
    c = case
    if c["kind"] == "train":
        return exact_train(c, seed)
    if c["kind"] == "predict":
        return exact_predict(c, seed)
    if work(c)["flops"] > 8.5e12:  # FP64 contractions of more than about 10 s
        return None
    key = 2503 * 10**6 + seed
    if c["kind"] == "batch":
        return [exact_counts(p, *network(p, sd, p["N"], p["M"]), key + i)
                for i, (p, sd) in enumerate(batch_parts(c, seed))]
    T, r = network(c, seed, c["N"], c["M"])
    which = dict(counts=exact_counts, moments=exact_moments, binned=exact_binned)[c["kind"]]
    return which(c, T, r, key)
