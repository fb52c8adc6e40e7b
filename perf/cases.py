"""Performance cases: the work that a user of the engine has it do, through its public entry points.

Each case is one call pattern of a program that samples the Holstein model: plain sweeps, learned
(cumulative) steps, exact weights of given configurations, mixed-shape groups and network training.
The model is the repository's own (t = M = Omega = 1, g = sqrt(2), half filling, dtau = 0.1); sizes
are those of its workloads (4x4 ... 16x16, beta up to 16, up to 256 chains) and of its tests (other
and unequal sides, restabilisation intervals that do not divide the number of slices).
"""
import math

import numpy as np
import torch

import paper_1905_07440_gb300 as hq
from workloads import HolsteinParams


# ------------------------------------------------------------------------------------ the cases

def listed():
    return [
        # one chain on a small lattice: a full sweep is a sequence of short dependent steps (latency)
        dict(name="sweep_4x4_one_chain", op="sweep", nx=4, ny=4, beta=4.0, n_wrap=10, chains=1, sites=0, local=True,
             block=True),
        # the batched workload: local moves and one block move per site, 256 chains
        dict(name="sweep_8x8_batched", op="sweep", nx=8, ny=8, beta=8.0, n_wrap=10, chains=256, sites=0, local=True,
             block=True),
        # largest lattice, local sweeps (how training configurations are made)
        dict(name="local_16x16", op="sweep", nx=16, ny=16, beta=16.0, n_wrap=10, chains=64, sites=0, local=True,
             block=False),
        # largest lattice, the reduced protocol's block moves (a run of sites)
        dict(name="blocks_16x16", op="sweep", nx=16, ny=16, beta=16.0, n_wrap=10, chains=64, sites=2, local=False,
             block=True),
        # learned sampler on the batched lattice: window of 20 slices and block moves, measured
        dict(name="learned_8x8_batched", op="learned", nx=8, ny=8, beta=8.0, n_wrap=10, chains=256, window=20,
             block=True, cnn=False),
        # the headline: learned sampler on the largest lattice, window of 32 slices, measured
        dict(name="learned_16x16", op="learned", nx=16, ny=16, beta=16.0, n_wrap=10, chains=64, window=32,
             block=False, cnn=False),
        # learned sampler whose block moves run on the convolutional action
        dict(name="learned_cnn_8x8", op="learned", nx=8, ny=8, beta=4.0, n_wrap=10, chains=64, window=20, block=True,
             cnn=True),
        # exact weights and G of given configurations (labels for training, checks), medium lattice
        dict(name="weight_12x12", op="weight", nx=12, ny=12, beta=8.0, n_wrap=10, chains=128),
        # the allocation-free log-determinant on a ragged shape (unequal sides, n_wrap does not divide L)
        dict(name="noalloc_10x6_ragged", op="noalloc", nx=10, ny=6, beta=3.3, n_wrap=7, chains=24),
        # engines of five shapes swept as one group
        dict(name="group_5_shapes", op="group", sides="4,6,8,10,12", betas="4,4,4,2,2", chains="64,64,48,32,16",
             n_wrap=10),
        # forward and backward pass of a training minibatch, patch network
        dict(name="gradient_patch_8x8", op="gradient", nx=8, ny=8, beta=8.0, n_wrap=10, batch=64, cnn=False),
        # the same for the convolutional action
        dict(name="gradient_cnn_8x8", op="gradient", nx=8, ny=8, beta=4.0, n_wrap=10, batch=32, cnn=True),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _side(rng, lo, hi):
    return 2 * rng.randint(lo // 2, hi // 2)


def _beta(rng, lo, hi):
    return _log_int(rng, int(10 * lo), int(10 * hi)) / 10.0


def draw(rng):
    """One more case of the same ranges, none dearer than the largest listed one."""
    most = max(_cost(c) for c in listed())
    while True:
        op = rng.choice(["sweep", "sweep", "sweep", "learned", "learned", "weight", "noalloc", "group", "gradient"])
        n_wrap = rng.choice([5, 7, 8, 10, 10, 10])
        if op == "sweep":
            local = rng.random() < 0.75
            nx, ny = _side(rng, 4, 16), _side(rng, 4, 16)
            c = dict(op=op, nx=nx, ny=ny, beta=_beta(rng, 1.0, 16.0), n_wrap=n_wrap, chains=_log_int(rng, 1, 256),
                     sites=rng.choice([0, 0, 1, 3, 8]), local=local, block=(not local) or rng.random() < 0.6)
        elif op == "learned":
            block = rng.random() < 0.5
            c = dict(op=op, nx=_side(rng, 4, 16), ny=_side(rng, 4, 16), beta=_beta(rng, 2.0, 16.0), n_wrap=n_wrap,
                     chains=_log_int(rng, 2, 256), window=rng.choice([0, 8, 20, 32]), block=block,
                     cnn=block and rng.random() < 0.3)
        elif op == "weight":
            c = dict(op=op, nx=_side(rng, 2, 16), ny=_side(rng, 2, 16), beta=_beta(rng, 1.0, 16.0), n_wrap=n_wrap,
                     chains=_log_int(rng, 1, 256))
        elif op == "noalloc":
            c = dict(op=op, nx=_side(rng, 2, 16), ny=_side(rng, 2, 16), beta=_beta(rng, 1.0, 16.0), n_wrap=n_wrap,
                     chains=_log_int(rng, 1, 292))
            if 7 * 8 * (c["nx"] * c["ny"]) ** 2 * c["chains"] > hq.NOALLOC_SCRATCH_BYTES:
                continue
        elif op == "group":
            k = rng.randint(2, 4)
            c = dict(op=op, sides=",".join(str(_side(rng, 4, 10)) for _ in range(k)),
                     betas=",".join(str(_beta(rng, 1.0, 4.0)) for _ in range(k)),
                     chains=",".join(str(_log_int(rng, 4, 64)) for _ in range(k)), n_wrap=n_wrap)
        else:
            c = dict(op=op, nx=_side(rng, 4, 12), ny=_side(rng, 4, 12), beta=_beta(rng, 2.0, 8.0), n_wrap=n_wrap,
                     batch=_log_int(rng, 8, 64), cnn=rng.random() < 0.4)
        if _cost(c) <= most:
            return c


# ---------------------------------------------------------------------------------- preparation

def _params(case, seed):
    return HolsteinParams(nx=case["nx"], ny=case["ny"], beta=case["beta"], n_wrap=case["n_wrap"],
                          seed=20190517 + int(seed))


def _fields(p, n, seed, ordered=False):
    """[n][L][N] start fields on the GPU: N(0, 1/(M Omega^2)) as the workloads draw them, or for the
    largest lattice at low temperature the charge-ordered start with the zero-point spread."""
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    X = torch.randn((n, p.n_slices, p.n_sites), dtype=torch.float64, device="cuda", generator=gen)
    if not ordered:
        return X
    i = torch.arange(p.n_sites, device="cuda")
    stag = 1.0 - 2.0 * ((i % p.nx + i // p.nx) % 2).double()
    return math.sqrt(0.5) * X - p.g + 0.9 * stag


def _patch_weights(p, seed):
    """Seeded weights of the patch network around the atomic limit, log|det| ~ sum dtau g |z| / 2
    (two hidden units carry z and -z of the centre), the rest random with a small output."""
    th = hq.init_network(int(seed), out_scale=0.3)
    w1, w2, w3 = th[:1600].reshape(25, 64), th[1664:5760].reshape(64, 64), th[5824:5888]
    w1[:, :2] = 0.0
    w1[10, 0], w1[10, 1] = 1.0, -1.0  # input 10: slice offset 0, the patch's own site
    w2[:2, :] = 0.0
    w2[:, :2] = 0.0
    w2[0, 0] = w2[1, 1] = 1.0
    w3[:2] = 0.4 * p.dtau * p.g
    return th


def prepare(case, seed):
    op = case["op"]
    if op == "group":
        engines = []
        for k, (side, beta, chains) in enumerate(_group(case)):
            p = HolsteinParams(nx=side, ny=side, beta=beta, n_wrap=case["n_wrap"], seed=20190517 + int(seed) + k)
            e = hq.Engine(p, chains)
            e.set_fields_device(_fields(p, chains, 1000 * int(seed) + k))
            engines.append(e)
        return dict(op=op, engines=engines, group=hq.Group(engines), out=[_host(e) for e in engines])
    p = _params(case, seed)
    if op == "noalloc":
        X = _fields(p, case["chains"], seed)
        return dict(op=op, p=p, X=X, out=torch.empty(case["chains"], dtype=torch.float64, device="cuda"))
    if op == "gradient":
        X = _fields(p, case["batch"], seed)
        gen = torch.Generator(device="cuda").manual_seed(int(seed) + 1)
        y = 5.0 * torch.randn(case["batch"], dtype=torch.float64, device="cuda", generator=gen)
        e = hq.Engine(p, 1)
        e.attach_network(case["batch"], case["batch"])
        if case["cnn"]:
            e.cnn_set_params(hq.init_cnn(seed, out_scale=0.3))
        else:
            e.set_params(hq.init_network(seed, out_scale=0.3))
        return dict(op=op, engine=e, X=X, y=y, cnn=case["cnn"])
    e = hq.Engine(p, case["chains"])
    if op == "weight":
        return dict(op=op, engine=e, X=_fields(p, case["chains"], seed))
    if op == "sweep":
        e.set_fields_device(_fields(p, case["chains"], seed))
        e.set_block_sites(case["sites"])
    else:
        e.set_fields_device(_fields(p, case["chains"], seed, ordered=True))
        e.attach_network(1, 1)
        e.set_params(_patch_weights(p, seed))
        if case["cnn"]:
            e.cnn_set_params(hq.init_cnn(seed, out_scale=0.03))
        e.set_inner_window(case["window"])
    return dict(op=op, engine=e, case=dict(case), out=_host(e))


def _host(e):
    """Page-locked buffer that receives the fields, as a sampling program keeps one."""
    return torch.empty(e.field_shape, dtype=torch.float64, pin_memory=True).numpy()


# -------------------------------------------------------------------------------------- one pass

def _read(e, out):
    """What a sampling program takes home after a step: fields, log-weights and electronic observables
    (the field averages follow from the fields; the wrap error is a rounding record, not a result)."""
    lw, ld = e.log_weight()
    obs = e.observables()
    r = dict(fields=e.get_fields(out), logw=lw, logdet=ld)
    for k in ("density", "double_occ", "s_cdw"):
        r[k] = np.array([o[k] for o in obs])
    for k in ("local_accepted", "global_accepted", "status"):
        r[k] = np.array([o[k] for o in obs], dtype=np.int64)
    return r


def run(state):
    op = state["op"]
    if op == "noalloc":
        stream = torch.cuda.current_stream().cuda_stream
        hq.logdet_noalloc(state["p"], state["X"], state["out"], stream=stream)
        return state["out"]
    if op == "group":
        state["group"].sweep(1)
        return [_read(e, o) for e, o in zip(state["engines"], state["out"])]
    e = state["engine"]
    if op == "gradient":
        grad, loss = (e.cnn_gradient if state["cnn"] else e.nn_gradient)(state["X"], state["y"])
        return dict(grad=grad, loss=loss)
    if op == "weight":
        e.set_fields_device(state["X"])
        lw, ld = e.log_weight()
        return dict(logw=lw, logdet=ld, green=e.green(0))
    c = state["case"]
    if op == "sweep":
        e.sweep(1, local=c["local"], global_=c["block"], measure=c["local"])
        return _read(e, state["out"])
    e.cumulative(1, 1, local=True, global_=c["block"], measure=True, cnn=c["cnn"])
    r = _read(e, state["out"])
    st = e.learned_stats()
    for k in ("inner_local_accepted", "inner_block_accepted", "cumulative_accepted"):
        r[k] = np.array([s[k] for s in st], dtype=np.int64)
    return r


# ------------------------------------------------------------------------------- algorithmic work

def _group(case):
    return [(int(s), float(b), int(c)) for s, b, c in zip(case["sides"].split(","), case["betas"].split(","),
                                                           case["chains"].split(","))]


def _chunks(L, w):
    return [min(w, L - s) for s in range(0, L, w)]


def _weight_flops(nx, ny, L, w, green=True):
    """Stabilised log|det M|: slice products through the separable propagator, QR, Q and the
    triangular factor per chunk, the final factorisation (and G)."""
    n = nx * ny
    f = 0.0
    for q, m in enumerate(_chunks(L, w)):
        f += m * (2.0 * n * n * (nx + ny) + n * n) + 8.0 / 3.0 * n ** 3 + (n ** 3 if q else 0.0)
    return f + (8.0 if green else 2.0) / 3.0 * n ** 3


def _local_flops(nx, ny, L, w):
    """Wraps and accepted moves (about 0.58) of every slice, a right factor and a fresh G per chunk."""
    n = nx * ny
    f = L * (4.0 * n * n * (nx + ny) + 2.0 * n * n + 0.58 * n * 2.0 * n * n)
    for m in _chunks(L, w):
        f += m * (2.0 * n * n * (nx + ny) + n * n) + (8.0 / 3.0 + 1.0 + 4.0 + 8.0 / 3.0) * n ** 3
    return f


def _block_flops(nx, ny, L, w):
    """One block move: the cheaper of the per-slice product and the chunk propagators."""
    n = nx * ny
    cm = 0.0
    for q, m in enumerate(_chunks(L, w)):
        cm += 2.0 * n ** 3 + 2.0 * m * n * n + m * m * (2.0 * n * (nx + ny) + n) + 8.0 / 3.0 * n ** 3
        cm += n ** 3 if q else 0.0
    return min(cm + 2.0 / 3.0 * n ** 3, _weight_flops(nx, ny, L, w, green=False))


PATCH = 2.0 * (25 * 64 + 64 * 64 + 64)       # one evaluation of the patch network
CONV = 2.0 * (27 * 16 + 27 * 256 + 27 * 16)  # one point of the convolutional action


def work(case):
    op = case["op"]
    if op == "group":
        r = dict(bytes=0.0, flops=0.0)
        for side, beta, chains in _group(case):
            one = work(dict(op="sweep", nx=side, ny=side, beta=beta, n_wrap=case["n_wrap"], chains=chains, sites=0,
                            local=True, block=True))
            r = {k: r[k] + one[k] for k in r}
        return r
    nx, ny, w = case["nx"], case["ny"], case["n_wrap"]
    n, L = nx * ny, int(round(case["beta"] / 0.1))
    if op == "gradient":
        points = float(case["batch"] * L * n)
        return dict(bytes=8.0 * points + 8.0 * case["batch"] + 4.0 * (hq.HQ_CNN_PARAMS if case["cnn"] else hq.HQ_NN_PARAMS),
                    flops=3.0 * points * (CONV if case["cnn"] else PATCH))
    C = case["chains"]
    if op in ("weight", "noalloc"):
        return dict(bytes=8.0 * C * (L * n + 1) + (8.0 * n * n if op == "weight" else 0.0),
                    flops=C * _weight_flops(nx, ny, L, w, green=op == "weight"))
    f = 0.0
    if op == "sweep":
        if case["local"]:
            f += _weight_flops(nx, ny, L, w) + _local_flops(nx, ny, L, w)
        if case["block"]:
            f += (min(case["sites"], n) or n) * _block_flops(nx, ny, L, w)
    else:
        slices = min(case["window"], L) or L
        f += _weight_flops(nx, ny, L, w) + slices * n * 25 * PATCH + L * n * PATCH
        if case["block"]:
            f += n * L * (9 * 2.0 * 27 * 16 + 25 * 2.0 * 27 * 256 + 49 * 2.0 * 27 * 16 if case["cnn"] else 5 * PATCH)
    return dict(bytes=16.0 * C * L * n, flops=C * f)


def _cost(case):
    """Rough seconds of a case, to keep the drawn ones below the listed ones: the FP64 work of the
    slowest chain on one SM or of all chains on the chip, whichever takes longer."""
    if case["op"] == "group":
        one = [_cost(dict(op="sweep", nx=s, ny=s, beta=b, n_wrap=case["n_wrap"], chains=1, sites=0, local=True,
                          block=True)) for s, b, _ in _group(case)]
        return max(max(one), sum(t * c for t, (_, _, c) in zip(one, _group(case))) / 152.0)
    f = work(case)["flops"]
    if case["op"] == "gradient":
        return f / 2e12
    return f / case["chains"] / 4e9 * max(1.0, case["chains"] / 152.0)


# ------------------------------------------------------------------- the same in plain 64 bits

def _hopping(nx, ny, dtau, sign):
    K = np.zeros((nx * ny, nx * ny))
    for y in range(ny):
        for x in range(nx):
            for dx, dy in ((1, 0), (-1, 0), (0, 1), (0, -1)):
                K[x + nx * y, (x + dx) % nx + nx * ((y + dy) % ny)] -= 1.0
    e, V = np.linalg.eigh(K)
    return (V * np.exp(-sign * dtau * e)) @ V.T


def _udv_green(p, X):
    """(G_0, log|det M|) of fields X [C][L][N] by column-sorted QR of the slice products."""
    E = torch.from_numpy(_hopping(p.nx, p.ny, p.dtau, 1.0))
    C, L, N = X.shape
    U = torch.eye(N, dtype=torch.float64).repeat(C, 1, 1)
    D = torch.ones(C, N, dtype=torch.float64)
    T = U.clone()
    V = torch.exp(-p.dtau * (p.g * X - p.mu))
    for s in range(0, L, 5):
        P = U * D[:, None, :]
        for l in range(s, min(s + 5, L)):
            P = E @ (V[:, l, :, None] * P)
        order = torch.argsort(torch.linalg.vector_norm(P, dim=1), dim=1, descending=True)
        U, R = torch.linalg.qr(torch.gather(P, 2, order[:, None, :].expand(C, N, N)))
        D = torch.diagonal(R, dim1=1, dim2=2).abs()
        T = (R / D[:, :, None]) @ torch.gather(T, 1, order[:, :, None].expand(C, N, N))
    big, small = D.clamp(min=1.0), D.clamp(max=1.0)
    rhs = U.transpose(1, 2) / big[:, :, None]
    A = rhs + small[:, :, None] * T
    return torch.linalg.solve(A, rhs), big.log().sum(1) + torch.linalg.slogdet(A)[1]


def _action(p, X):
    kin = ((torch.roll(X, -1, 1) - X) ** 2).sum((1, 2))
    return p.mass / (2.0 * p.dtau) * kin + 0.5 * p.dtau * p.mass * p.omega ** 2 * (X ** 2).sum((1, 2))


def _uniforms(seed, chain, sweep, event, tag):
    """Two uniforms of one Philox4x32-10 block."""
    m = 0xFFFFFFFF
    c0, c1, c2, c3, k0, k1 = event, sweep, chain, tag, seed & m, (seed >> 32) & m
    for _ in range(10):
        a, b = 0xD2511F53 * c0, 0xCD9E8D57 * c2
        c0, c1, c2, c3 = (b >> 32) ^ c1 ^ k0, b & m, (a >> 32) ^ c3 ^ k1, a & m
        k0, k1 = (k0 + 0x9E3779B9) & m, (k1 + 0xBB67AE85) & m
    return tuple(((x >> 5) * 67108864 + (y >> 6)) / 9007199254740992.0 for x, y in ((c0, c1), (c2, c3)))


def _plain_chain(p, X, case, chain):
    """One sweep of one chain, move by move, every G and determinant from the fields."""
    L, N = X.shape
    n_loc = n_blk = 0
    E, Ei = _hopping(p.nx, p.ny, p.dtau, 1.0), _hopping(p.nx, p.ny, p.dtau, -1.0)
    stag = np.array([1.0 - 2.0 * ((i % p.nx + i // p.nx) % 2) for i in range(N)])
    obs = []
    fresh = lambda Y: [t[0].numpy() for t in _udv_green(p, torch.from_numpy(Y)[None])]  # noqa: E731
    if case["local"]:
        G = fresh(X)[0]
        for l in range(L):
            for i in range(N):
                u1, u2 = _uniforms(p.seed, chain, 0, l * N + i, 0)
                x, xp, xm = X[l, i], X[(l + 1) % L, i], X[l - 1, i]
                y = x + p.dx_local * (2.0 * u1 - 1.0)
                dS = p.mass / (2.0 * p.dtau) * ((xp - y) ** 2 + (y - xm) ** 2 - (xp - x) ** 2 - (x - xm) ** 2)
                dS += 0.5 * p.dtau * p.mass * p.omega ** 2 * (y * y - x * x)
                delta = math.exp(-p.dtau * p.g * (p.dx_local * (2.0 * u1 - 1.0))) - 1.0
                R = 1.0 + delta * (1.0 - G[i, i])
                if u2 < R * R * math.exp(-dS):
                    col = G[:, i].copy()
                    col[i] -= 1.0
                    G = G + delta / R * np.outer(col, G[i, :])
                    X[l, i] = y
                    n_loc += 1
            d = np.exp(-p.dtau * (p.g * X[l] - p.mu))
            G = E @ (d[:, None] * G / d[None, :]) @ Ei
            if (l + 1) % p.n_wrap == 0 or l + 1 == L:
                G = fresh(np.roll(X, -(l + 1), axis=0))[0]
                m = 1.0 - np.diag(G)
                scdw = 4.0 * (stag @ m) ** 2 + 2.0 * np.trace(G) - 2.0 * stag @ (G * G.T) @ stag
                obs.append((2.0 * m.mean(), (m * m).mean(), scdw / N))
    ld = float(fresh(X)[1])
    if case["block"]:
        sites = range(N)
        if 0 < case["sites"] < N:
            j0 = min(int(_uniforms(p.seed, chain, 0, N, 1)[0] * N), N - 1)
            sites = [(j0 + k) % N for k in range(case["sites"])]
        for i in sites:
            u1, u2 = _uniforms(p.seed, chain, 0, i, 1)
            dx = p.dx_global * (2.0 * u1 - 1.0)
            Y = X.copy()
            Y[:, i] += dx
            new = float(fresh(Y)[1])
            dS = 0.5 * p.dtau * p.mass * p.omega ** 2 * float(((X[:, i] + dx) ** 2 - X[:, i] ** 2).sum())
            if u2 < math.exp(min(2.0 * (new - ld) - dS, 709.0)):
                X, ld = Y, new
                n_blk += 1
    return X, ld, np.array(obs).mean(0) if obs else np.full(3, np.nan), n_loc, n_blk


def _exact_gradient(case, X, y, theta):
    """Loss and gradient of the mean squared error with the bfloat16 weights, in 64 bits."""
    th = torch.from_numpy(theta).bfloat16().double().requires_grad_()
    nx, ny, L, B = case["nx"], case["ny"], X.shape[1], X.shape[0]
    z = (X.cpu() + math.sqrt(2.0)).reshape(B, L, ny, nx)
    y = y.cpu()
    loss = torch.zeros((), dtype=torch.float64)
    for a in range(B):
        v = z[a]
        if case["cnn"]:
            w1, b1, w2, b2, w3, b3 = torch.split(th, [432, 16, 6912, 16, 432, 1])
            w1 = w1.reshape(3, 3, 3, 1, 16).permute(4, 3, 0, 1, 2)
            w2 = w2.reshape(3, 3, 3, 16, 16).permute(4, 3, 0, 1, 2)
            w3 = w3.reshape(3, 3, 3, 16, 1).permute(4, 3, 0, 1, 2)
            h = v[None, None]
            for k, (w, b) in enumerate(((w1, b1), (w2, b2), (w3, b3))):
                h = torch.nn.functional.pad(h, (1, 1, 1, 1, 1, 1), mode="circular")
                h = torch.nn.functional.conv3d(h, w, b)
                h = torch.relu(h) if k < 2 else h
        else:
            w1, b1, w2, b2, w3, b3 = torch.split(th, [1600, 64, 4096, 64, 64, 1])
            cross = [(0, 0), (1, 0), (-1, 0), (0, 1), (0, -1)]
            rows = [torch.roll(v, (-dl, -dy, -dx), (0, 1, 2)).reshape(-1) for dl in range(-2, 3) for dx, dy in cross]
            h = torch.relu(torch.stack(rows, 1) @ w1.reshape(25, 64) + b1)
            h = torch.relu(h @ w2.reshape(64, 64) + b2) @ w3 + b3
        one = (h.sum() - y[a]) ** 2 / B
        one.backward()
        loss += one.detach()
    return dict(grad=th.grad.numpy(), loss=float(loss))


def exact(case, seed):
    op = case["op"]
    if op in ("group", "learned"):
        # a network-driven chain is a sequence of single-precision decisions; a group runs hundreds of
        # full chain-sweeps (minutes move by move)
        return None
    p = _params(case, seed)
    if op == "gradient":
        if work(case)["flops"] > 2.5e11:
            return None
        s = prepare(case, seed)
        theta = (hq.init_cnn if case["cnn"] else hq.init_network)(seed, out_scale=0.3)
        return _exact_gradient(case, s["X"], s["y"], theta)
    X = _fields(p, case["chains"], seed).cpu()
    if op in ("weight", "noalloc"):
        if case["chains"] * p.n_slices * p.n_sites ** 3 > 4e10:
            return None
        G, ld = _udv_green(p, X)
        if op == "noalloc":
            return ld
        return dict(logw=2.0 * ld - _action(p, X), logdet=ld, green=G[0])
    moves = (p.n_wrap if case["local"] else 0) + ((min(case["sites"], p.n_sites) or p.n_sites) if case["block"] else 0)
    if case["chains"] * p.n_slices * (moves * p.n_sites ** 2 * 2e-8 + moves * 4e-5 + p.n_sites * 5e-5) > 10.0:
        return None
    ends = [_plain_chain(p, X[c].numpy().copy(), case, c) for c in range(case["chains"])]
    F = torch.from_numpy(np.stack([r[0] for r in ends]))
    ld = torch.tensor([r[1] for r in ends], dtype=torch.float64)
    obs = np.stack([r[2] for r in ends])
    return dict(fields=F, logw=2.0 * ld - _action(p, F), logdet=ld, density=obs[:, 0], double_occ=obs[:, 1],
                s_cdw=obs[:, 2], local_accepted=np.array([r[3] for r in ends]),
                global_accepted=np.array([r[4] for r in ends]), status=np.zeros(len(ends), dtype=np.int64))
