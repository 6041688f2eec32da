"""What is measured on a GPU: the work a user of this framework has it do,
through its public entry points, over the range of sizes that it serves.

Each case is one call, or one short chain of calls, on inputs that are already
where such a program has them (device tensors; host arrays for the request
server).  Sizes are those of the repository's own workloads (the paper's CPD,
Kronecker-compression, tensor-regression and serving settings) and the ranges
around them.  Results are checked against ``exact``: the same definition
evaluated in 64 bits with torch, hash tables included.
"""
from __future__ import annotations

import math
import random
import weakref

import numpy as np
import torch

import paper_2106_13062_gb300 as fcs

DEV = "cuda"

# ------------------------------------------------------------------ cases


def listed():
    """The listed cases (see the comment at each for what it stands for)."""
    return [
        # the smallest call: one CP sketch of a 20^3 rank-5 tensor from a seed
        # (a program that sketches many tiny tensors pays this per tensor)
        dict(name="cp_tiny", kind="cp", I="20,20,20", J="8,8,8", R=5, D=1),
        # an ordinary, ragged order-4 CP sketch (FFT length 8192)
        dict(name="cp_ragged", kind="cp", I="310,77,523,151", J="700,1900,450,1300", R=37, D=5),
        # CP-form FCS at scale, the repository's headline (FFT length 16384)
        dict(name="cp_scale", kind="cp", I="1000,1000,1000", J="5000,5000,5000", R=100, D=10),
        # the upper end of the serving mix: order 4, rank 256, FFT length 32768
        dict(name="cp_long", kind="cp", I="2000,1500,900,1203", J="8192,8000,7001,6000", R=256,
             D=10),
        # dense-route sketch of the robust tensor power method's tensor (one
        # per deflated tensor, the largest single read of the framework)
        dict(name="dense_rtpm", kind="dense", shape="500,500,500", J="2000,2000,2000", D=5, nb=1,
             perm="C"),
        # one RTPM step's contractions: T(u,u,u) and T(I,u,u) of 64 vectors
        dict(name="contract_rtpm", kind="contract", what="both", I="500,500,500",
             J="2000,2000,2000", D=5, B=64, m=0),
        # Kronecker compression of 32 pairs of 512 x 512 matrices: two batched
        # dense sketches and the outer combine
        dict(name="kron_compress", kind="kron", pairs=32, n=512, J=1024, D=10),
        # decompression: 2^20 sampled entries of each of the 32 products
        dict(name="kron_recover", kind="recover", pairs=32, I="512,512,512,512",
             J="1024,1024,1024,1024", D=10, M=1 << 20),
        # 64 uneven CP problems in one planned launch chain (the batch layer
        # under the request server)
        dict(name="batch_mixed", kind="batch", count=64, shapes=5),
        # a whole sketched CP-ALS run: three sweeps on a 400^3 sketch, rank 10
        dict(name="als_400", kind="als", I="400,400,400", J="3000,3000,3000", R=10, D=3, sweeps=3),
        # forward pass of a compressed tensor regression layer: sketch a batch
        # of 7 x 7 x 32 activations, inner products with 10 class weights
        dict(name="trl_forward", kind="trl", shape="7,7,32", J=60, D=5, B=256, C=10),
        # a burst of mixed requests to the server (host arrays in and out)
        dict(name="serve_burst", kind="serve", count=48, shapes=70),
    ]


_KINDS = ("cp", "dense", "contract", "kron", "recover", "batch", "als", "trl", "serve")


def _logi(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _s(v):
    return ",".join(str(int(x)) for x in v)


def _l(text):
    return [int(x) for x in str(text).split(",")]


def draw(rng):
    """One more case of the same ranges: a kind, and sizes spread over its range."""
    kind = rng.choice(_KINDS)
    if kind == "cp":
        N = rng.choice((2, 3, 3, 4))
        return dict(kind=kind, I=_s(_logi(rng, 20, 2000) for _ in range(N)),
                    J=_s(_logi(rng, 8, 8192) for _ in range(N)), R=_logi(rng, 1, 256),
                    D=rng.randint(1, 10))
    if kind == "dense":
        N = rng.choice((2, 3, 3, 4))
        D = rng.randint(1, 10)
        total = math.exp(rng.uniform(math.log(1e3), math.log(6e8 / D / 5)))
        w = [rng.uniform(0.7, 1.3) for _ in range(N)]
        shape = [max(2, int(total ** (x / sum(w)))) for x in w]
        nb = _logi(rng, 1, max(1, min(32, int(6e8 / D / math.prod(shape)))))
        return dict(kind=kind, shape=_s(shape), J=_s(_logi(rng, 8, 4096) for _ in range(N)), D=D,
                    nb=nb, perm=rng.choice(("C", "C", "F")))
    if kind == "contract":
        N = rng.choice((3, 3, 4))
        return dict(kind=kind, what=rng.choice(("both", "all", "free")),
                    I=_s(_logi(rng, 50, 500) for _ in range(N)),
                    J=_s(_logi(rng, 256, 4096) for _ in range(N)), D=rng.randint(1, 10),
                    B=_logi(rng, 1, 64), m=rng.randrange(N))
    if kind == "kron":
        return dict(kind=kind, pairs=rng.randint(1, 32), n=_logi(rng, 16, 512),
                    J=_logi(rng, 64, 1024), D=rng.randint(1, 10))
    if kind == "recover":
        N = rng.choice((2, 3, 4, 4))
        return dict(kind=kind, pairs=rng.randint(1, 32), I=_s(_logi(rng, 16, 512) for _ in range(N)),
                    J=_s(_logi(rng, 64, 2000) for _ in range(N)), D=rng.randint(1, 10),
                    M=_logi(rng, 1000, 1 << 20))
    if kind == "batch":
        c = dict(kind=kind, count=rng.randint(2, 56), shapes=rng.randrange(10, 1 << 20))
        while c["count"] > 2 and work(c)["flops"] > 3e10:
            c["count"] -= 1
        return c
    if kind == "als":
        return dict(kind=kind, I=_s(_logi(rng, 50, 400) for _ in range(3)),
                    J=_s(_logi(rng, 1000, 4096) for _ in range(3)), R=rng.randint(2, 10),
                    D=rng.randint(1, 5), sweeps=rng.randint(1, 3))
    if kind == "trl":
        return dict(kind=kind, shape=_s((rng.randint(3, 14), rng.randint(3, 14), rng.randint(8, 64))),
                    J=_logi(rng, 16, 400), D=rng.randint(1, 7), B=_logi(rng, 1, 1024),
                    C=_logi(rng, 2, 200))
    c = dict(kind=kind, count=rng.randint(2, 40), shapes=rng.randrange(10, 1 << 20))
    while c["count"] > 2 and work(c)["flops"] > 1.2e10:
        c["count"] -= 1
    return c


def _jt(J):
    return sum(J) - len(J) + 1


def _plen(Jt):
    return 1 << max(4, (Jt - 1).bit_length())


def _mixed_shapes(seed, count):
    """Uneven CP problems of the serving mix: order 3-4, I log-U[50, 2000], R
    log-U[1, 256], J log-U[256, 8192], D U{1..10}."""
    rng = random.Random(1000 + seed)
    out = []
    for _ in range(count):
        N = rng.randint(3, 4)
        out.append(([_logi(rng, 50, 2000) for _ in range(N)], [_logi(rng, 256, 8192) for _ in range(N)],
                    _logi(rng, 1, 256), rng.randint(1, 10)))
    return out


def _burst(seed, count):
    """Requests of a burst: about half CP sketches of the serving mix, half
    contractions of 1-16 vectors with one of four resident sketches."""
    rng = random.Random(2000 + seed)
    resident = []
    for _ in range(4):
        i, j = rng.randint(50, 499), rng.randint(256, 1999)
        resident.append(([i] * 3, [j] * 3, 8, 5))
    shapes = _mixed_shapes(seed, count)
    reqs = []
    for k in range(count):
        if rng.random() < 0.5:
            reqs.append(("cp", shapes[k]))
        else:
            reqs.append(("ct", rng.randrange(4), rng.random() < 0.5, rng.randint(1, 16)))
    return resident, reqs


# ------------------------------------------------------------------ inputs
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device=DEV, dtype=torch.float32)


def _weights(g, R):
    return torch.rand(R, generator=g, device=DEV) + 0.5


def _cp_inputs(g, I, R):
    return [_randn(g, i, R) for i in I], _weights(g, R)


def _unit(g, B, I):
    u = _randn(g, B, I)
    return u / u.norm(dim=1, keepdim=True)


def _dense_input(c, seed):
    """A low-rank tensor with noise, as CPD meets it; perm F: the first mode is
    the contiguous one (a tensor from a column-major program)."""
    shape, nb = _l(c["shape"]), c["nb"]
    g = _gen(seed)
    lay = shape[::-1] if c["perm"] == "F" else shape
    T = _randn(g, nb, *lay) * 0.01
    rest = math.prod(lay[1:])
    for b in range(nb):
        a, w = _randn(g, lay[0], 4), _randn(g, 4, rest)
        T[b].view(lay[0], rest).add_((a @ w) * (1.0 / math.sqrt(rest)))
    if c["perm"] == "F":
        T = T.permute(0, *range(len(shape), 0, -1))
    return T


_ctx = None


def _context():
    """The one context that a program keeps."""
    global _ctx
    if _ctx is None:
        _ctx = fcs.Context()
    return _ctx


_server = None


def _srv():
    """The one request server that a program keeps."""
    global _server
    if _server is None:
        _server = fcs.FcsServer(device=torch.cuda.current_device(), streams=4, max_inflight=128,
                                max_batch=48, arena_bytes=6 << 30, staging_bytes=1 << 30)
    return _server


def prepare(case, seed):
    """Inputs of `seed` on the GPU (host arrays for the server), and the
    context, plan or server a program keeps."""
    c, kind, ctx = case, case["kind"], _context()
    g = _gen(seed)
    st = {"c": c, "ctx": ctx, "seed": seed}
    if kind == "cp":
        st["U"], st["lam"] = _cp_inputs(g, _l(c["I"]), c["R"])
        st["J"] = _l(c["J"])
    elif kind == "dense":
        st["T"], st["J"] = _dense_input(c, seed), _l(c["J"])
        st["h"], st["s"] = fcs.fcs_make_hashes(ctx, seed, _l(c["shape"]), st["J"], c["D"])
    elif kind == "contract":
        I, J = _l(c["I"]), _l(c["J"])
        st["I"], st["J"] = I, J
        st["h"], st["s"] = fcs.fcs_make_hashes(ctx, seed, I, J, c["D"])
        U, lam = _cp_inputs(g, I, 10)
        U = [u / math.sqrt(u.shape[0]) for u in U]
        st["T"] = _cp64(U, lam, J, *_split(I, st["h"], st["s"])).float()
        st["v"] = [_unit(g, c["B"], i) for i in I]
    elif kind == "kron":
        n = c["n"]
        st["A"], st["B"] = _randn(g, c["pairs"], n, n), _randn(g, c["pairs"], n, n)
        st["J"] = [c["J"]] * 4
        st["h"], st["s"] = fcs.fcs_make_hashes(ctx, seed, [n] * 4, st["J"], c["D"])
    elif kind == "recover":
        I, J = _l(c["I"]), _l(c["J"])
        st["I"], st["J"] = I, J
        st["h"], st["s"] = fcs.fcs_make_hashes(ctx, seed, I, J, c["D"])
        st["sk"] = _randn(g, c["pairs"], c["D"], _jt(J))
        st["idx"] = torch.stack([torch.randint(0, i, (c["pairs"], c["M"]), generator=g, device=DEV,
                                               dtype=torch.int32) for i in I], dim=2).contiguous()
    elif kind == "batch":
        probs, st["keep"] = [], []
        for k, (I, J, R, D) in enumerate(_mixed_shapes(c["shapes"], c["count"])):
            U, lam = _cp_inputs(g, I, R)
            h, s = fcs.fcs_make_hashes(ctx, seed * 64 + k, I, J, D)
            pr, out = fcs.cp_problem(U, lam, J, h, s)
            probs.append(pr)
            st["keep"].append((U, lam, h, s, out))
        st["plan"] = fcs.BatchPlan(ctx, probs)
    elif kind == "als":
        I, J, R = _l(c["I"]), _l(c["J"]), c["R"]
        st["I"], st["J"] = I, J
        st["h"], st["s"] = fcs.fcs_make_hashes(ctx, seed, I, J, c["D"])
        U, lam = _cp_inputs(g, I, R)
        st["T"] = _cp64(U, lam, J, *_split(I, st["h"], st["s"])).float()
        st["F"] = [(u + 0.3 * _randn(g, *u.shape)).t().contiguous() for u in U]
    elif kind == "trl":
        shape = _l(c["shape"])
        st["J"] = [c["J"]] * 3
        st["h"], st["s"] = fcs.fcs_make_hashes(ctx, seed, shape, st["J"], c["D"])
        st["X"] = torch.relu(_randn(g, c["B"], *shape))
        W = _randn(g, c["C"], *shape) / math.sqrt(math.prod(shape))
        st["sw"] = _dense64(W, st["J"], *_split(shape, st["h"], st["s"])).float()
        st["bias"] = _randn(g, c["C"])
    else:
        return _serve_prepare(c, seed)
    return st


class _Served:
    """Host data of one burst and the resident sketches it contracts with."""

    def __init__(self, c, seed):
        self.srv, self.seed = _srv(), seed
        resident, reqs = _burst(c["shapes"], c["count"])
        g = np.random.default_rng(seed)
        self.resident, self.sids = resident, []
        tickets = []
        for k, (I, J, R, D) in enumerate(resident):
            U = [g.standard_normal((i, R), dtype=np.float32) for i in I]
            lam = g.uniform(0.5, 1.5, R).astype(np.float32)
            self.resident[k] = (I, J, R, D, U, lam)
            tickets.append(self.srv.submit_cp(U, lam, J, D, seed=seed + k, keep_resident=True))
        self.sids = [self.srv.wait(t).sketch_id for t in tickets]
        self.reqs = []
        for r in reqs:
            if r[0] == "cp":
                I, J, R, D = r[1]
                U = [g.standard_normal((i, R), dtype=np.float32) for i in I]
                lam = g.uniform(0.5, 1.5, R).astype(np.float32)
                self.reqs.append(("cp", I, J, R, D, U, lam))
            else:
                I = resident[r[1]][0]
                v = [g.standard_normal((r[3], i), dtype=np.float32) for i in I]
                v = [x / np.linalg.norm(x, axis=1, keepdims=True) for x in v]
                self.reqs.append(("ct", r[1], r[2], v))
        weakref.finalize(self, _Served._release, self.srv, list(self.sids))

    @staticmethod
    def _release(srv, sids):
        for s in sids:
            srv.release(s)


def _serve_prepare(c, seed):
    return {"c": c, "served": _Served(c, seed)}


# ------------------------------------------------------------------ one pass
def run(st):
    """One pass through the public entry points; its outputs, whole."""
    c = st["c"]
    kind = c["kind"]
    if kind == "serve":
        return _serve_run(st["served"])
    ctx, J = st["ctx"], st.get("J")
    if kind == "cp":
        out, h, s = fcs.fcs_sketch_cp_seeded(ctx, st["U"], st["lam"], J, c["D"], st["seed"])
        return {"sketch": out, "h": h, "s": s}
    if kind == "dense":
        if c["nb"] == 1:
            return fcs.fcs_sketch_dense(ctx, st["T"][0], J, st["h"], st["s"])
        return fcs.fcs_sketch_dense(ctx, st["T"], J, st["h"], st["s"], batched=True)
    if kind == "contract":
        if c["what"] == "both":
            return fcs.fcs_contract_both(ctx, st["T"], st["v"], st["I"], J, st["h"], st["s"],
                                         free_mode=c["m"])
        k = fcs.FCS_CONTRACT_ALL if c["what"] == "all" else fcs.FCS_CONTRACT_FREE
        return fcs.fcs_contract(ctx, k, st["T"], st["v"], st["I"], J, st["h"], st["s"],
                                free_mode=c["m"])
    if kind == "kron":
        n2, ld = 2 * c["n"], 4 * c["n"]
        fa = fcs.fcs_sketch_dense(ctx, st["A"], J[:2], st["h"][:, :n2], st["s"][:, :n2], ldh=ld,
                                  batched=True)
        fb = fcs.fcs_sketch_dense(ctx, st["B"], J[2:], st["h"][:, n2:], st["s"][:, n2:], ldh=ld,
                                  batched=True)
        return fcs.fcs_sketch_outer(ctx, fa, fb)
    if kind == "recover":
        return fcs.fcs_recover(ctx, st["sk"], st["I"], J, st["h"], st["s"], st["idx"])
    if kind == "batch":
        st["plan"].launch()
        return [k[4] for k in st["keep"]]
    if kind == "als":
        F = [f.clone() for f in st["F"]]
        lam = fcs.fcs_als(ctx, st["T"], st["I"], J, st["h"], st["s"], F, c["sweeps"])
        return {"lam": lam, "F": F}
    sa = fcs.fcs_sketch_dense(ctx, st["X"], J, st["h"], st["s"], batched=True)
    return fcs.fcs_sketch_inner(ctx, sa, st["sw"], st["bias"])


def _serve_run(sv):
    srv, tickets, outs = sv.srv, [], []
    for k, r in enumerate(sv.reqs):
        if r[0] == "cp":
            _, I, J, R, D, U, lam = r
            out = np.empty((D, _jt(J)), dtype=np.float32)
            tickets.append(srv.submit_cp(U, lam, J, D, seed=sv.seed + 100 + k, out=out))
        else:
            _, q, every, v = r
            I, J = sv.resident[q][0], sv.resident[q][1]
            if every:
                out = np.empty((v[0].shape[0],), dtype=np.float32)
                tickets.append(srv.submit_contract(sv.sids[q], I, J, fcs.FCS_CONTRACT_ALL, v, out))
            else:
                out = np.empty((v[0].shape[0], I[0]), dtype=np.float32)
                tickets.append(srv.submit_contract(sv.sids[q], I, J, fcs.FCS_CONTRACT_FREE,
                                                   [None, v[1], v[2]], out, free_mode=0))
        outs.append(out)
    for t in tickets:
        if srv.wait(t).state != 2:
            raise RuntimeError("a served request failed")
    return outs


# ------------------------------------------------------------------ work
def _fft(P):
    return 2.5 * P * math.log2(P)          # one real FFT of length P


def _cp_work(I, J, R, D):
    N, Jt = len(I), _jt(J)
    P = _plen(Jt)
    return dict(bytes=4 * (sum(I) * R + R) + 5 * D * sum(I) + 4 * D * Jt,
                flops=D * (N * R + 1) * _fft(P) + D * R * (P / 2 + 1) * (6 * (N - 1) + 2))


def _contract_work(what, I, J, D, B, m):
    N, Jt = len(I), _jt(J)
    P = _plen(Jt)
    nvec = N - 1 if what == "free" else N
    vec = sum(I) - (I[m] if what == "free" else 0)
    ffts = D + B * D * (nvec + (0 if what == "all" else 1))
    out = (B if what != "free" else 0) + (B * I[m] if what != "all" else 0)
    return dict(bytes=4 * (D * Jt + B * vec + out) + 5 * D * sum(I),
                flops=ffts * _fft(P) + B * D * (P / 2 + 1) * 6 * (nvec + 1))


def _add(*w):
    return dict(bytes=sum(x["bytes"] for x in w), flops=sum(x["flops"] for x in w))


def work(case):
    """Bytes (inputs read once, outputs written once) and algorithmic
    operations of one pass."""
    c, kind = case, case["kind"]
    if kind == "cp":
        I, J = _l(c["I"]), _l(c["J"])
        return _cp_work(I, J, c["R"], c["D"])
    if kind == "dense":
        I, J = _l(c["shape"]), _l(c["J"])
        n = math.prod(I) * c["nb"]
        return dict(bytes=4 * n + 5 * c["D"] * sum(I) + 4 * c["nb"] * c["D"] * _jt(J),
                    flops=c["D"] * n)
    if kind == "contract":
        return _contract_work(c["what"], _l(c["I"]), _l(c["J"]), c["D"], c["B"], c["m"])
    if kind == "kron":
        J, D, n, p = [c["J"]] * 4, c["D"], c["n"], c["pairs"]
        P = _plen(_jt(J))
        return dict(bytes=8 * p * n * n + 20 * D * n + 4 * p * D * _jt(J),
                    flops=2 * p * D * n * n + p * D * (3 * _fft(P) + 3 * P))
    if kind == "recover":
        I, J = _l(c["I"]), _l(c["J"])
        n = c["pairs"] * c["M"]
        return dict(bytes=4 * n * (len(I) + 1) + 4 * c["pairs"] * c["D"] * _jt(J) + 5 * c["D"] * sum(I),
                    flops=n * c["D"] * len(I))
    if kind == "batch":
        return _add(*[_cp_work(*x) for x in _mixed_shapes(c["shapes"], c["count"])])
    if kind == "als":
        I, J, R, D = _l(c["I"]), _l(c["J"]), c["R"], c["D"]
        one = [_contract_work("free", I, J, D, R, m) for m in range(len(I))]
        fl = c["sweeps"] * sum(w["flops"] for w in one) + \
            c["sweeps"] * sum(4 * R * R * sum(I) for _ in I)
        return dict(bytes=4 * D * _jt(J) + 5 * D * sum(I) + 8 * R * sum(I) + 4 * R, flops=fl)
    if kind == "trl":
        I, J, D = _l(c["shape"]), [c["J"]] * 3, c["D"]
        n = math.prod(I)
        return dict(bytes=4 * c["B"] * n + 5 * D * sum(I) + 4 * c["C"] * D * _jt(J) + 4 * c["C"] +
                    4 * c["B"] * c["C"], flops=c["B"] * D * n + 2 * c["B"] * c["C"] * D * _jt(J))
    resident, reqs = _burst(c["shapes"], c["count"])
    ws = []
    for r in reqs:
        if r[0] == "cp":
            ws.append(_cp_work(*r[1]))
        else:
            I, J, _, D = resident[r[1]]
            ws.append(_contract_work("all" if r[2] else "free", I, J, D, r[3], 0))
    return _add(*ws)


# ------------------------------------------------------------------ 64 bits
_P61 = (1 << 61) - 1
_M64 = (1 << 64) - 1


def _mix(seed, k):
    z = (seed + (k + 1) * 0x9E3779B97F4A7C15) & _M64
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & _M64
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & _M64
    return z ^ (z >> 31)


def _hashes(seed, I, J, D):
    """The hash family in Python integers: Carter-Wegman over 2^61 - 1, four
    SplitMix64 draws per (sketch, mode).  h and s, [D][mode] int64 tensors."""
    H, S = [], []
    for d in range(D):
        hr, sr = [], []
        for n, (i_n, j_n) in enumerate(zip(I, J)):
            k = 4 * (d * len(I) + n)
            ah, bh = 1 + _mix(seed, k) % (_P61 - 1), _mix(seed, k + 1) % _P61
            as_, bs = 1 + _mix(seed, k + 2) % (_P61 - 1), _mix(seed, k + 3) % _P61
            hr.append(torch.tensor([(ah * i + bh) % _P61 % j_n for i in range(i_n)], device=DEV))
            sr.append(torch.tensor([1 - 2 * (((as_ * i + bs) % _P61) & 1) for i in range(i_n)],
                                   device=DEV))
        H.append(hr)
        S.append(sr)
    return H, S


def _split(I, h, s):
    """The tables [D, sum I] that a call returned, as [D][mode] tensors."""
    return [list(r.split(I)) for r in h.long()], [list(r.split(I)) for r in s]


def _cs(h, s, X, P):
    """Count Sketch of the rows of X ([B, I], 64 bits) in P bins."""
    out = torch.zeros(X.shape[0], P, dtype=torch.float64, device=DEV)
    return out.index_add_(1, h, X * s.double())


def _cp64(U, lam, J, H, S):
    Jt = _jt(J)
    P = _plen(Jt)
    R, step = U[0].shape[1], max(1, (1 << 25) // P)
    rows = []
    for d in range(len(H)):
        acc = torch.zeros(P // 2 + 1, dtype=torch.complex128, device=DEV)
        for r in range(0, R, step):
            p = lam[r:r + step].double()[:, None].to(torch.complex128)
            for n, u in enumerate(U):
                p = p * torch.fft.rfft(_cs(H[d][n], S[d][n], u[:, r:r + step].double().t(), P))
            acc += p.sum(0)
        rows.append(torch.fft.irfft(acc, P)[:Jt])
    return torch.stack(rows)


def _dense64(T, J, H, S, modes=None):
    """[nb, D, Jt] of a batch of tensors T (any strides)."""
    shape = list(T.shape[1:])
    modes = list(range(len(shape))) if modes is None else modes
    rows = math.prod(shape[:-1])
    out = torch.zeros(T.shape[0], len(H), _jt(J), dtype=torch.float64, device=DEV)
    flat = T.reshape(T.shape[0], rows, shape[-1])
    step = max(1, (1 << 23) // shape[-1])
    for d in range(len(H)):
        hl, sl = H[d][modes[0]], S[d][modes[0]]
        for n in modes[1:-1]:
            hl = (hl[:, None] + H[d][n][None, :]).reshape(-1)
            sl = (sl[:, None] * S[d][n][None, :]).reshape(-1)
        if len(modes) == 1:
            hl, sl = torch.zeros(1, dtype=torch.int64, device=DEV), torch.ones(1, dtype=torch.int64, device=DEV)
        hz, sz = H[d][modes[-1]], S[d][modes[-1]]
        for r in range(0, rows, step):
            idx = (hl[r:r + step, None] + hz[None, :]).reshape(-1)
            sg = (sl[r:r + step, None] * sz[None, :]).double()
            for b in range(T.shape[0]):
                out[b, d].index_add_(0, idx, (flat[b, r:r + step].double() * sg).reshape(-1))
    return out


def _median(x, dim):
    v = x.sort(dim=dim).values
    D = x.shape[dim]
    a, b = v.select(dim, (D - 1) // 2), v.select(dim, D // 2)
    return 0.5 * (a + b)


def _spectra64(T, P):
    return torch.fft.rfft(T.double(), P)


def _contract64(spec, v, J, H, S, P, what, m):
    """Medians over the sketches of T(v..v) and T(v, I, v)."""
    al, fr = [], []
    for d in range(spec.shape[0]):
        F = [None if x is None else torch.fft.rfft(_cs(H[d][n], S[d][n], x.double(), P))
             for n, x in enumerate(v)]
        if what != "free":
            q = spec[d].conj()[None, :]
            for f in F:
                q = q * f
            w = torch.full((P // 2 + 1,), 2.0, dtype=torch.float64, device=DEV)
            w[0] = w[-1] = 1.0
            al.append((q.real * w).sum(1) / P)
        if what != "all":
            q = spec[d][None, :]
            for n, f in enumerate(F):
                if n != m:
                    q = q * f.conj()
            z = torch.fft.irfft(q, P)
            fr.append(z[:, H[d][m]] * S[d][m].double())
    return (_median(torch.stack(al, 1), 1) if al else None,
            _median(torch.stack(fr, 1), 1) if fr else None)


def exact(case, seed):
    """What run() returns for these inputs, evaluated in 64 bits with torch."""
    c, kind = case, case["kind"]
    if kind == "serve":
        return _serve_exact(prepare(case, seed)["served"])
    st = prepare(case, seed)
    J = st.get("J")
    if kind == "cp":
        I = _l(c["I"])
        H, S = _hashes(seed, I, J, c["D"])
        cat = lambda rows, t: torch.stack([torch.cat(r) for r in rows]).to(t)  # noqa: E731
        return {"sketch": _cp64(st["U"], st["lam"], J, H, S), "h": cat(H, torch.int32),
                "s": cat(S, torch.int8)}
    if kind == "dense":
        out = _dense64(st["T"], J, *_hashes(seed, _l(c["shape"]), J, c["D"]))
        return out[0] if c["nb"] == 1 else out
    if kind == "contract":
        I, P = st["I"], _plen(_jt(J))
        H, S = _hashes(seed, I, J, c["D"])
        al, fr = _contract64(_spectra64(st["T"], P), st["v"], J, H, S, P, c["what"], c["m"])
        return (al, fr) if c["what"] == "both" else al if c["what"] == "all" else fr
    if kind == "kron":
        H, S = _hashes(seed, [c["n"]] * 4, J, c["D"])
        a = _dense64(st["A"], J[:2], H, S, modes=[0, 1])
        b = _dense64(st["B"], J[2:], H, S, modes=[2, 3])
        P = _plen(_jt(J))
        return torch.fft.irfft(torch.fft.rfft(a, P) * torch.fft.rfft(b, P), P)[..., :_jt(J)].contiguous()
    if kind == "recover":
        H, S = _hashes(seed, st["I"], J, c["D"])
        out = torch.empty(c["pairs"], c["M"], dtype=torch.float64, device=DEV)
        for p in range(c["pairs"]):
            ix = st["idx"][p].long()
            raw = []
            for d in range(c["D"]):
                hs = sum(H[d][n][ix[:, n]] for n in range(len(J)))
                sg = math.prod([S[d][n][ix[:, n]] for n in range(len(J))])
                raw.append(st["sk"][p, d].double()[hs] * sg)
            out[p] = _median(torch.stack(raw), 0)
        return out
    if kind == "batch":
        outs = []
        for k, ((I, J, R, D), (U, lam, *_)) in enumerate(zip(_mixed_shapes(c["shapes"], c["count"]),
                                                            st["keep"])):
            outs.append(_cp64(U, lam, J, *_hashes(seed * 64 + k, I, J, D)))
        return outs
    if kind == "als":
        I, P = st["I"], _plen(_jt(J))
        H, S = _hashes(seed, I, J, c["D"])
        spec, F = _spectra64(st["T"], P), [f.double() for f in st["F"]]
        lam = None
        for _ in range(c["sweeps"]):
            for m in range(len(I)):
                v = [None if n == m else F[n] for n in range(len(I))]
                M = _contract64(spec, v, J, H, S, P, "free", m)[1]
                G = torch.ones(c["R"], c["R"], dtype=torch.float64, device=DEV)
                for n in range(len(I)):
                    if n != m:
                        G = G * (F[n] @ F[n].t())
                X = torch.linalg.solve(G, M)
                lam = X.norm(dim=1)
                F[m] = X / lam[:, None]
        return {"lam": lam, "F": F}
    sa = _dense64(st["X"], J, *_hashes(seed, _l(c["shape"]), J, c["D"]))
    return _median(torch.einsum("bdj,cdj->bcd", sa, st["sw"].double()), 2) + st["bias"].double()


def _serve_exact(sv):
    cu = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(DEV)  # noqa: E731
    T64, HS = [], []
    for k, (I, J, R, D, U, lam) in enumerate(sv.resident):
        HS.append(_hashes(sv.seed + k, I, J, D))
        T64.append(_spectra64(_cp64([cu(u) for u in U], cu(lam), J, *HS[k]), _plen(_jt(J))))
    outs = []
    for k, r in enumerate(sv.reqs):
        if r[0] == "cp":
            _, I, J, R, D, U, lam = r
            o = _cp64([cu(u) for u in U], cu(lam), J, *_hashes(sv.seed + 100 + k, I, J, D))
        else:
            _, q, every, v = r
            J = sv.resident[q][1]
            al, fr = _contract64(T64[q], [cu(x) for x in v], J, *HS[q], _plen(_jt(J)),
                                 "all" if every else "free", 0)
            o = al if every else fr
        outs.append(o.cpu().numpy())
    return outs
