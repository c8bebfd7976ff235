"""The work that users of the library have it do, as cases that can be timed.

Every case goes through the public entry points (binding.CRF, binding.Server,
unrolled.unrolled_log_marginals).  A case's "kind" says which:

  grid      mean-field solve of a batch of 4- or 8-connected grids
  frame     the same for a new image: unaries and edge weights are set first,
            so the step-size constant is computed too
  dense     fully connected Gaussian CRF
  sparse    general graph from an edge list
  unrolled  one training step through K unrolled steps (loss gradient
            included, outputs log q and the three gradients)
  serve     a burst of requests through the continuous-batching server

Sizes follow the repository's benchmark (64 x 64 binary denoising, 512 x 512
segmentation with 21 labels, 96 x 96 fully connected, the serving mix, the
16 x 256 x 256 unrolled batch, the two edge-list graphs) and odd ones around
them.  "eta": 0 asks the library for its own step size.
"""
import math

import numpy as np
import torch

from paper_1511_06103_gb300 import binding
from paper_1511_06103_gb300.unrolled import unrolled_log_marginals

DEV = "cuda"
OFFSETS = ((0, 1), (1, 0), (1, 1), (1, -1))   # right, down, down-right, down-left
RULES = {"fixed": binding.MF_RULE_FIXED, "momentum": binding.MF_RULE_MOMENTUM, "adhoc": binding.MF_RULE_ADHOC}


def listed():
    return [
        # binary denoising of one small image: a whole solve is one short launch,
        # and the caller reads F at the end
        dict(name="denoise_64", kind="grid", B=1, H=64, W=64, L=2, conn=4, sym=True, bf16=False, rule="fixed",
             iters=50, eta=0.0, rel_tol=0.0, energy=True),
        # a few small odd images with an asymmetric compatibility
        dict(name="small_batch_ragged", kind="grid", B=5, H=61, W=45, L=7, conn=8, sym=False, bf16=False,
             rule="fixed", iters=20, eta=safe_eta(8, 7), rel_tol=0.0, energy=False),
        # the benchmark's segmentation solve, model resident on the device
        dict(name="seg_512", kind="grid", B=1, H=512, W=512, L=21, conn=8, sym=True, bf16=False, rule="fixed",
             iters=100, eta=0.0, rel_tol=0.0, energy=False),
        # a new photograph of an odd size, all the way from unaries to marginals
        dict(name="seg_frame_375x500", kind="frame", B=1, H=375, W=500, L=21, conn=8, sym=True, bf16=False,
             rule="fixed", iters=100, eta=0.0, rel_tol=0.0, energy=True),
        # a batch of odd images with more labels, stopping rule on
        dict(name="seg_batch_27", kind="grid", B=4, H=333, W=479, L=27, conn=8, sym=True, bf16=False, rule="fixed",
             iters=40, eta=safe_eta(8, 27), rel_tol=1e-9, energy=False),
        # many labels with tensor-core messages and two FP32 refinement steps
        dict(name="seg_bf16_32", kind="grid", B=1, H=512, W=512, L=32, conn=8, sym=True, bf16=True, rule="fixed",
             iters=98, eta=safe_eta(8, 32), rel_tol=0.0, energy=False),
        # the benchmark's fully connected model, both precisions
        dict(name="dense_f32", kind="dense", B=1, H=96, W=96, L=21, bf16=False, fly=False, iters=30),
        dict(name="dense_bf16", kind="dense", B=1, H=96, W=96, L=21, bf16=True, fly=False, iters=28),
        # edge lists: a large random graph, and the layers of a belief network
        dict(name="sparse_random", kind="sparse", N=262144, deg=4, L=21, layers=False, sym=True, iters=50),
        dict(name="sparse_layers", kind="sparse", N=12288, deg=64, L=2, layers=True, sym=True, iters=100),
        # one training step of the benchmark's unrolled batch
        dict(name="unrolled_train", kind="unrolled", B=16, H=256, W=256, L=21, conn=4, sym=True, K=10, eta=0.05),
        # the serving mix arriving at once (more of it than the small end of a quiet minute)
        dict(name="serve_burst", kind="serve", n=28, lo=64, hi=512, iters=60, per_step=4),
    ]


def safe_eta(conn, L):
    """A step below 1/(1 + curvature) for random compatibilities with entries in (-1, 1)."""
    return 1.0 / (1.0 + 1.2 * conn * math.sqrt(L))


def _log(rng, lo, hi):
    return max(lo, min(hi, round(math.exp(rng.uniform(math.log(lo), math.log(hi))))))


def draw(rng):
    kind = rng.choices(["grid", "frame", "dense", "sparse", "unrolled", "serve"], [9, 3, 4, 3, 4, 2])[0]
    conn, sym, L = rng.choice([4, 8]), rng.random() < 0.75, rng.choice([2, 8, 21, rng.randint(2, 32)])
    if kind in ("grid", "frame"):
        H, W, B = _log(rng, 24, 640), _log(rng, 24, 640), rng.choice([1, 1, 2, rng.randint(2, 8)])
        bf16 = kind == "grid" and L >= 16 and rng.random() < 0.4
        rule = "fixed" if bf16 or kind == "frame" or rng.random() < 0.8 else rng.choice(["momentum", "adhoc"])
        iters = rng.choice([10, 20, 50, 100])
        while B > 1 and B * H * W * L * iters > 512 * 512 * 21 * 100:
            B -= 1
        while iters > 10 and B * H * W * L * iters > 512 * 512 * 21 * 100:
            iters //= 2
        own = kind == "frame" and sym
        tol = 1e-9 if kind == "grid" and L >= 8 and not bf16 and rng.random() < 0.3 else 0.0
        return dict(kind=kind, B=B, H=H, W=W, L=L, conn=conn, sym=sym, bf16=bf16, rule=rule, iters=iters,
                    eta=0.0 if own else safe_eta(conn, L), rel_tol=tol, energy=rng.random() < 0.3)
    if kind == "dense":
        bf16 = rng.random() < 0.5
        return dict(kind=kind, B=rng.choice([1, 1, 2]), H=_log(rng, 16, 96), W=_log(rng, 16, 96), L=min(L, 24),
                    bf16=bf16, fly=bf16 and rng.random() < 0.4, iters=rng.choice([5, 10, 28]))
    if kind == "sparse":
        layers = rng.random() < 0.4
        N = _log(rng, 600, 20000 if layers else 262144)
        return dict(kind=kind, N=N, deg=rng.choice([16, 64]) if layers else rng.randint(1, 6), L=min(L, 24),
                    layers=layers, sym=sym, iters=rng.choice([10, 30, 50]))
    if kind == "unrolled":
        H, W, L, K = _log(rng, 24, 256), _log(rng, 24, 256), min(L, 24), rng.randint(2, 10)
        B = rng.randint(1, 16)
        while B > 1 and B * H * W * L * L * (conn + 4) * (1 if sym else 2) * K > 16 * 256 * 256 * 21 * 21 * 8 * 10:
            B -= 1
        return dict(kind=kind, B=B, H=H, W=W, L=L, conn=conn, sym=sym, K=K, eta=min(0.05, safe_eta(conn, L)))
    return dict(kind=kind, n=rng.randint(3, 24), lo=rng.choice([32, 64]), hi=_log(rng, 96, 480),
                iters=rng.choice([20, 40, 60]), per_step=rng.choice([1, 4]))


# ---- inputs ------------------------------------------------------------------

def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _smooth(B, C, H, W, g):
    """[B][C][H][W] smooth fields in [0, 1]: uniform noise on an 8-pixel lattice, interpolated."""
    low = torch.rand((B, C, H // 8 + 2, W // 8 + 2), generator=g, device=DEV)
    f = torch.nn.functional.interpolate(low, size=(H, W), mode="bicubic", align_corners=True)
    lo, hi = f.amin((2, 3), keepdim=True), f.amax((2, 3), keepdim=True)
    return (f - lo) / (hi - lo)


def _edge(t, dy, dx):
    """The two ends of the edges (y, x) -> (y+dy, x+dx) of a [..., H, W] or [..., H, W, L] array as index pairs."""
    H, W = t
    a = (slice(0, H - dy), slice(max(0, -dx), W - max(0, dx)))
    b = (slice(dy, H), slice(max(0, dx), W + min(0, dx)))
    return a, b


def _weights(B, H, W, conn, g):
    """w = exp(-|dc|^2 / (2 * 0.1^2)) over a smooth colour field, zero where the edge leaves the image."""
    rgb = _smooth(B, 3, H, W, g)
    w = torch.zeros((B, conn // 2, H, W), device=DEV)
    for k in range(conn // 2):
        a, b = _edge((H, W), *OFFSETS[k])
        w[(slice(None), k) + a] = torch.exp(
            -(rgb[(slice(None),) * 2 + a] - rgb[(slice(None),) * 2 + b]).square().sum(1) / 0.02)
    return w


def _mu(L, sym, g):
    m = torch.rand((L, L), generator=g, device=DEV) * 2 - 1
    if sym:
        m = torch.triu(m, 1)
        m = m + m.T
    return m.contiguous()


def _unary(shape, g):
    return -torch.log_softmax(2.0 * torch.randn(shape, generator=g, device=DEV), -1)


def _denoise(B, H, W, g):
    """Noisy binary images: blobs with a fifth of the pixels flipped; unaries are the flip costs."""
    clean = _smooth(B, 1, H, W, g).reshape(B, H * W) > 0.5
    noisy = clean ^ (torch.rand((B, H * W), generator=g, device=DEV) < 0.2)
    hit, miss = -math.log(0.8), -math.log(0.2)
    return torch.where(torch.stack([~noisy, noisy], -1), hit, miss).float().contiguous()


def _inputs(case, seed):
    """The arrays of a case (device tensors; the requests of a server are host arrays)."""
    g, c = _gen(seed), case
    if c["kind"] in ("grid", "frame", "unrolled"):
        B, H, W, L = c["B"], c["H"], c["W"], c["L"]
        if L == 2 and c["conn"] == 4 and c["sym"]:
            U, mu = _denoise(B, H, W, g), 0.8 * (1 - torch.eye(2, device=DEV))
        else:
            U, mu = _unary((B, H * W, L), g), _mu(L, c["sym"], g)
        d = dict(U=U, mu=mu, w=_weights(B, H, W, c["conn"], g))
        if c["kind"] == "unrolled":
            d["y"] = _smooth(B, L, H, W, g).argmax(1).reshape(B, H * W)
        return d
    if c["kind"] == "dense":
        B, H, W, L = c["B"], c["H"], c["W"], c["L"]
        y, x = torch.meshgrid(torch.arange(H, device=DEV), torch.arange(W, device=DEV), indexing="ij")
        pos = torch.stack([x, y], -1).reshape(1, H * W, 2).float().expand(B, -1, -1)
        rgb = 255.0 * _smooth(B, 3, H, W, g).reshape(B, 3, H * W).transpose(1, 2)
        return dict(U=_unary((B, H * W, L), g), mu=(1 - torch.eye(L, device=DEV)) + 0.5 * _mu(L, True, g),
                    feats=torch.cat([pos, rgb], -1).contiguous(), theta=(3.0, 13.0))
    if c["kind"] == "sparse":
        N, L = c["N"], c["L"]
        if c["layers"]:   # a third of the variables on top, each joined to `deg` of those below
            top = N // 3
            src = torch.arange(top, device=DEV).repeat_interleave(c["deg"])
            dst = top + torch.randint(0, N - top, src.shape, generator=g, device=DEV)
        else:
            src = torch.randint(0, N, (N * c["deg"],), generator=g, device=DEV)
            dst = (src + torch.randint(1, N, src.shape, generator=g, device=DEV)) % N
        w = 0.2 + 0.8 * torch.rand(src.shape, generator=g, device=DEV)
        return dict(U=_unary((N, L), g), mu=(0.3 if c["layers"] else 1.0) * _mu(L, c["sym"], g),
                    src=src.int(), dst=dst.int(), w=w)
    reqs = []   # serve: square images, sides spread over the range, label counts taken in turn
    for i in range(c["n"]):
        side = round(c["lo"] * (c["hi"] / c["lo"]) ** ((i * 7 % c["n"] + 0.5) / c["n"]))
        L = (2, 8, 21)[i % 3]
        one = _inputs(dict(kind="grid", B=1, H=side, W=side, L=L, conn=4 if L == 2 else 8, sym=True), seed * 1000 + i)
        reqs.append(dict(H=side, W=side, conn=4 if L == 2 else 8, tol=0.0 if L == 2 else 1e-9,
                         U=one["U"][0].cpu().numpy(), mu=one["mu"].cpu().numpy(), w=one["w"][0].cpu().numpy()))
    return dict(reqs=reqs)


# ---- one pass ------------------------------------------------------------------

def prepare(case, seed):
    d, c = _inputs(case, seed), case
    kind = c["kind"]
    if kind == "unrolled":
        for k in ("U", "mu", "w"):
            d[k].requires_grad_(True)
        return dict(case=c, d=d)
    if kind == "serve":
        return dict(case=c, d=d, srv=binding.Server(2 << 30, max_slots=128))
    if kind == "sparse":
        crf = binding.CRF(binding.CRF_SPARSE, c["L"], 1, c["N"])
        crf.set_graph(d["mu"].cpu().numpy(), d["src"].cpu().numpy(), d["dst"].cpu().numpy(), d["w"].cpu().numpy())
        crf.set_unary(d["U"])
    elif kind == "dense":
        crf = binding.CRF(binding.CRF_DENSE_GAUSS, c["L"], c["H"], c["W"], batch=c["B"],
                          precision=binding.CRF_BF16 if c["bf16"] else binding.CRF_FP32)
        crf.set_unary(d["U"])
        crf.set_pairwise(d["mu"], d["feats"], theta=d["theta"])
        if c["fly"]:
            crf.dense_on_the_fly(True)
    else:
        crf = binding.CRF(binding.CRF_GRID8 if c["conn"] == 8 else binding.CRF_GRID4, c["L"], c["H"], c["W"],
                          batch=c["B"], precision=binding.CRF_BF16 if c["bf16"] else binding.CRF_FP32)
        if kind == "grid":
            crf.set_unary(d["U"])
            crf.set_pairwise(d["mu"], d["w"])
    q = torch.empty((crf.B, crf.N, crf.L), device=DEV)
    return dict(case=c, d=d, crf=crf, q=q)


def run(state):
    c, d = state["case"], state["d"]
    kind = c["kind"]
    if kind == "serve":
        srv = state["srv"]
        left = [srv.submit(r["U"], r["mu"], r["w"], r["H"], r["W"], r["conn"], eta=0.0, max_iters=c["iters"],
                           rel_tol=r["tol"]) for r in d["reqs"]]
        got = {}
        while left:
            srv.step(c["per_step"])
            wait = []
            for t in left:
                st, _, _, q = srv.poll(t)
                if st == 2:
                    got[t] = q
                else:
                    wait.append(t)
            left = wait
        return [got[t] for t in sorted(got)]
    if kind == "unrolled":
        logq = unrolled_log_marginals(d["U"], d["mu"], d["w"], c["H"], c["W"], c["conn"], c["K"], c["eta"])
        loss = torch.nn.functional.nll_loss(logq.reshape(-1, c["L"]), d["y"].reshape(-1))
        return [logq.detach(), *torch.autograd.grad(loss, (d["U"], d["mu"], d["w"]))]
    crf, q = state["crf"], state["q"]
    if kind == "frame":
        crf.set_unary(d["U"])
        crf.set_pairwise(d["mu"], d["w"])
    refine = 2 if c.get("bf16") else 0
    energy = c.get("energy", False)
    crf.iterate(c["iters"], eta=c.get("eta", 0.0), reset=True, rel_tol=c.get("rel_tol", 0.0), refine_fp32=refine,
                final_free_energy=energy, rule=RULES[c.get("rule", "fixed")])
    crf.marginals(q)
    # F goes into a float32 log: the steps and the messages in it are FP32
    return [q, crf.free_energy().astype(np.float32)] if energy else [q]


def work(case):
    """Inputs read once, outputs written once, and the arithmetic of every step."""
    c = case
    kind = c["kind"]
    if kind == "serve":
        tot = dict(bytes=0.0, flops=0.0)
        for i in range(c["n"]):
            side = round(c["lo"] * (c["hi"] / c["lo"]) ** ((i * 7 % c["n"] + 0.5) / c["n"]))
            L = (2, 8, 21)[i % 3]
            one = work(dict(kind="grid", B=1, H=side, W=side, L=L, conn=4 if L == 2 else 8, sym=True,
                            iters=c["iters"]))
            tot = {k: tot[k] + one[k] for k in tot}
        return tot
    L = c["L"]
    per_var = 12 * L   # update, softmax, free energy
    if kind in ("grid", "frame"):
        n = c["B"] * c["H"] * c["W"]
        msg = 2 * c["conn"] * L + 2 * L * L * (1 if c["sym"] else 2)
        return dict(bytes=4.0 * n * (2 * L + c["conn"] // 2), flops=float(n) * c["iters"] * (msg + per_var))
    if kind == "dense":
        N = c["H"] * c["W"]
        return dict(bytes=4.0 * c["B"] * N * (2 * L + 5),
                    flops=float(c["B"]) * c["iters"] * N * (2.0 * N * L + 2 * L * L + per_var))
    if kind == "sparse":
        N = c["N"]
        E = (N // 3 if c["layers"] else N) * c["deg"]
        return dict(bytes=4.0 * (2 * N * L + 3 * E),
                    flops=float(c["iters"]) * (4.0 * E * L + N * (2 * L * L * (1 if c["sym"] else 2) + per_var)))
    n = c["B"] * c["H"] * c["W"]   # unrolled: forward, then the products for d/dq, d/dmu and d/dw
    msg = 2 * c["conn"] * L + 2 * L * L * (1 if c["sym"] else 2)
    return dict(bytes=4.0 * n * (3 * L + c["conn"]) + 8.0 * n, flops=float(n) * c["K"] * (4 * msg + 3 * per_var))


# ---- the same in 64 bits ---------------------------------------------------------

def _grid_sums(q, w, conn):
    """(sum over edges leaving, sum over edges entering) of w times the other end's q; q [B][H][W][L]."""
    So, Si = torch.zeros_like(q), torch.zeros_like(q)
    for k in range(conn // 2):
        a, b = _edge(q.shape[1:3], *OFFSETS[k])
        a, b = (slice(None),) + a, (slice(None),) + b
        wk = w[:, k][a][..., None]
        So[a] = So[a] + wk * q[b]
        Si[b] = Si[b] + wk * q[a]
    return So, Si


def _top_eigenvalue(op, shape, centre=False):
    """Largest eigenvalue of a symmetric operator (Lanczos, 64 bits), on centred rows if asked."""
    g = _gen(7)
    v = torch.randn(shape, generator=g, device=DEV, dtype=torch.float64)
    if centre:
        v = v - v.mean(-1, keepdim=True)
    v, old, b, al, be = v / v.norm(), torch.zeros_like(v), 0.0, [], []
    for _ in range(min(500, v.numel() - 1)):
        u = op(v) - b * old
        al.append(torch.sum(u * v))
        u = u - al[-1] * v
        b = u.norm()
        if len(al) % 50 == 0 and float(b) < 1e-10:
            break
        be.append(b)
        old, v = v, u / b
    al, be = torch.stack(al).cpu().numpy(), torch.stack(be).cpu().numpy()[: len(al) - 1]
    T = np.diag(al) + np.diag(be, 1) + np.diag(be, -1)
    return float(np.linalg.eigvalsh(T[np.ix_(np.isfinite(al), np.isfinite(al))])[-1])


def _solve(U, message, eta, iters, rule="fixed", s=None):
    """log q after `iters` parallel steps from softmax(-U), and F of it."""
    s = torch.log_softmax(-U, -1) if s is None else s
    avg = None
    for _ in range(iters):
        q = torch.exp(s)
        grad = U + message(q)
        if rule == "adhoc":
            s = torch.log((1 - eta) * q + eta * torch.softmax(-grad, -1))
            continue
        if rule == "momentum":
            avg = grad if avg is None else 0.95 * avg + (1 - 0.95) * grad
            grad = avg
        s = torch.log_softmax((1 - eta) * s - eta * grad, -1)
    return s


def _energy(U, message, s):
    q = torch.exp(s)
    return (q * (U + 0.5 * message(q) + s)).flatten(1).sum(1)


def _grid_message(mu, w, conn):
    def message(q):
        B, _, H, W = w.shape
        So, Si = _grid_sums(q.reshape(B, H, W, -1), w, conn)
        return (So @ mu.T + Si @ mu).reshape(q.shape)
    return message


def exact(case, seed):
    d, c = _inputs(case, seed), case
    kind = c["kind"]
    if kind == "serve":
        out = []
        for r in d["reqs"]:
            U, mu, w = (torch.from_numpy(r[k]).to(DEV).double() for k in ("U", "mu", "w"))
            So, Si = _grid_sums(torch.ones((1, r["H"], r["W"], 1), device=DEV, dtype=torch.float64), w[None], r["conn"])
            eta = 1 / (1 + float((So + Si).max()) * _mu_extreme(mu))
            s = _solve(U[None], _grid_message(mu, w[None], r["conn"]), eta, c["iters"])
            out.append(torch.exp(s)[0])
        return out
    if kind == "unrolled":
        U, mu, w = (d[k].double().requires_grad_(True) for k in ("U", "mu", "w"))
        s = _solve(U, _grid_message(mu, w, c["conn"]), c["eta"], c["K"])
        loss = torch.nn.functional.nll_loss(s.reshape(-1, c["L"]), d["y"].reshape(-1))
        return [s.detach(), *torch.autograd.grad(loss, (U, mu, w))]
    U, mu = d["U"].double(), d["mu"].double()
    if kind == "sparse":
        src, dst, w = d["src"].long(), d["dst"].long(), d["w"].double()[:, None]
        out_of = torch.sparse_coo_tensor(torch.stack([src, dst]), w[:, 0], (c["N"],) * 2).coalesce().to_sparse_csr()
        into = torch.sparse_coo_tensor(torch.stack([dst, src]), w[:, 0], (c["N"],) * 2).coalesce().to_sparse_csr()

        def message(q):
            return (out_of @ q[0] @ mu.T + into @ q[0] @ mu)[None]
        one = torch.ones((c["N"], 1), device=DEV, dtype=torch.float64)
        D = (float((out_of @ one + into @ one).max()) * _mu_extreme(mu) if c["sym"] else
             (float((out_of @ one).max()) + float((into @ one).max())) * float(mu.norm()))
        return [torch.exp(_solve(U[None], message, 1 / (1 + D), c["iters"]))]
    if kind == "dense":
        sp, sc = (1 / (math.sqrt(2) * t) for t in d["theta"])
        K = []
        for b in range(c["B"]):
            f = d["feats"][b].double() * torch.tensor([sp, sp, sc, sc, sc], device=DEV, dtype=torch.float64)
            K.append(torch.exp(-torch.cdist(f, f, compute_mode="donot_use_mm_for_euclid_dist").square()).fill_diagonal_(0))
        K = torch.stack(K)
        eta = torch.tensor([_own_eta(lambda v, b=b: K[b] @ v, lambda v, b=b: K[b] @ v @ mu, K.shape[1], mu)
                            for b in range(c["B"])], device=DEV, dtype=torch.float64)[:, None, None]
        return [torch.exp(_solve(U, lambda q: K @ q @ mu, eta, c["iters"] + (2 if c["bf16"] else 0)))]
    w = d["w"].double()
    message = _grid_message(mu, w, c["conn"])
    eta = c["eta"]
    if eta <= 0:
        B, _, H, W = w.shape

        def adjacency(b):
            return lambda v: sum(_grid_sums(v.reshape(1, H, W, 1), w[b:b + 1], c["conn"])).reshape(H * W, 1)
        eta = torch.tensor([_own_eta(adjacency(b), _grid_message(mu, w[b:b + 1], c["conn"]), H * W, mu)
                            for b in range(B)], device=DEV, dtype=torch.float64)[:, None, None]
    s = _solve(U, message, eta, c["iters"] + (2 if c["bf16"] else 0), c["rule"])
    return [torch.exp(s), _energy(U, message, s)] if c["energy"] else [torch.exp(s)]


def _mu_spectrum(mu):
    C = torch.eye(len(mu), device=DEV, dtype=torch.float64) - 1 / len(mu)
    return torch.linalg.eigvalsh(C @ ((mu + mu.T) / 2) @ C)


def _mu_extreme(mu):
    return float(_mu_spectrum(mu).abs().max())


def _own_eta(adjacency, message, N, mu):
    """1 / (1 + max(Lambda, 0)), Lambda the curvature on the tangent space of the simplices; for symmetric mu it is
    the largest product of an eigenvalue of the edge weights and one of the centred mu."""
    if torch.equal(mu, mu.T):
        top = _top_eigenvalue(adjacency, (N, 1))
        low = -_top_eigenvalue(lambda v: -adjacency(v), (N, 1))
        nu = _mu_spectrum(mu)
        lam = max(top * float(nu[-1]), top * float(nu[0]), low * float(nu[-1]), low * float(nu[0]))
    else:
        def centred(v):
            m = message(v[None])[0]
            return m - m.mean(-1, keepdim=True)
        lam = _top_eigenvalue(centred, (N, len(mu)), centre=True)
    return 1 / (1 + max(lam, 0.0))
