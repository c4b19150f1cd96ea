"""Cases of the BSE Haydock library: what its users' programs call, at the sizes they call it with.

Every case goes through `paper_1602_01863_gb300.bse`, as `bench.py`, the
training loop of the learned residual and the tests do.  Sizes are those of
the repository's own workloads (`synth.py`, `bench.py`, the tests): coarse
meshes of 3^3 to 12^3 points refined 2 to 4 times per axis, 2 to 6 valence and
conduction bands, 1 to 4 vectors.

Kinds: "apply" (one H application), "haydock" (a recursion of some steps on a
handle that is kept), "batch" (many systems in one graph launch), "spectrum_run"
(a new system from the model to its spectrum, set-up included), "gradients"
(the residual network's training pass) and "pairs" (its training data).

With FP32 vectors the Lanczos coefficients carry FP32 precision, although the
library hands them out in 64-bit arrays: those runs return them as float32.
"""
import math

import numpy as np
import torch

from paper_1602_01863_gb300 import bse, synth

PREC = {"f64": bse.PREC_F64, "f32": bse.PREC_F32, "bf16": bse.PREC_BF16}
SCHEME = {"m1": bse.SCHEME_M1, "m2": bse.SCHEME_M2, "m3": bse.SCHEME_M3}
ETA = synth.ETA
WIDTH = 128                      # hidden width of the residual network


def _system(name, kind, n, nd, nv, nc, vecs, scheme, kc, **more):
    c = dict(kind=kind, n=n, nd=nd, nv=nv, nc=nc, vecs=vecs, scheme=scheme, kc=kc, **more)
    return dict(name=name, **c) if name else c


def listed():
    return [
        # the smallest call: one H application of the small configuration in the FP64 plain path (a solver of the user's own
        # that calls H itself); latency and launches count
        _system("apply_small_f64", "apply", 4, 2, 3, 3, 1, "m3", "f64", width=1.0),
        # the small configuration's Haydock run with full reorthogonalisation, as the parity and width studies run it
        _system("haydock_small_f64_cgs2", "haydock", 4, 2, 3, 3, 1, "m3", "f64", width=1.0, steps=100, cgs2=True),
        # Method 2 (the stored dense H) on the small configuration, three polarisations
        _system("haydock_m2_f64", "haydock", 4, 2, 3, 3, 3, "m2", "f64", width=1.0, steps=40, cgs2=False),
        # a ragged system without tensor-core storage: odd bands, odd meshes, four vectors, a wider near region
        _system("apply_ragged_c64", "apply", 7, 3, 3, 5, 4, "m3", "f32", width=1.5),
        # K_c and dense tables from elsewhere (another crystal's, as from an ab initio code) on the mixed path
        _system("apply_caller_tables", "apply", 6, 4, 4, 4, 3, "m3", "bf16", width=1.0, caller=True),
        # the benchmark's system in the FP64 plain path: one H application to three vectors
        _system("apply_single_f64", "apply", 8, 4, 4, 4, 3, "m3", "f64", width=1.0),
        # the benchmark's system on the mixed path: the Haydock step loop itself, three polarisations
        _system("haydock_single_mixed", "haydock", 8, 4, 4, 4, 3, "m3", "bf16", width=1.0, steps=24, cgs2=False),
        # the same from nothing: a user with a new system pays for K_c, the tables and the first run too
        _system("spectrum_single_mixed", "spectrum_run", 8, 4, 4, 4, 3, "m3", "bf16", width=1.0, steps=24, cgs2=False),
        # the uneven batch of 24 systems (72 chains) as one graph launch
        dict(name="batch_24_mixed", kind="batch", first=100, count=24, steps=12),
        # the largest system: Method 1 with the learned near-diagonal residual, three vectors
        _system("apply_largest_learned", "apply", 12, 4, 4, 6, 3, "m1", "bf16", width=1.0, learned=8),
        # one training pass of the residual network at the training loop's batch
        dict(name="gradients_4096", kind="gradients", bands=24, rows=4096),
        # training data for it: 512 sampled dense pairs of a coarse 4^3 system, every band pair
        _system("pairs_512", "pairs", 4, 4, 4, 6, 1, "m1", "f32", width=1.0, blocks=512),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["apply", "apply", "apply", "haydock", "haydock", "spectrum_run", "batch", "gradients", "pairs"])
    if kind == "gradients":
        return dict(kind=kind, bands=rng.choice([4, 6, 9, 12, 15, 16, 20, 24]), rows=log_int(100, 4096))
    if kind == "batch":
        return dict(kind=kind, first=rng.randrange(100, 124), count=log_int(3, 16), steps=rng.randint(6, 12))
    nv, nc = rng.randint(2, 4), rng.randint(2, 6)
    if kind == "pairs":
        return _system("", kind, rng.choice([3, 4, 5]), rng.choice([2, 3, 4]), nv, nc, 1, "m1", rng.choice(["f32", "f64"]),
                       width=1.0, blocks=log_int(50, 512))
    kc = rng.choice(["bf16", "bf16", "f32", "f64"])
    scheme = rng.choice(["m1", "m3", "m3"])
    n, nd = rng.randint(3, 6 if kc == "f64" else 8), rng.randint(2, 4)
    if kind == "spectrum_run":                  # a production system: the spectrum itself is what counts
        n, nv, nc = rng.randint(7, 8), rng.randint(3, 4), rng.randint(3, 5)
        kc = "bf16" if kc == "f64" else kc
    more = {"width": 1.0 if n < 4 else rng.choice([0.5, 1.0, 1.0, 1.5])}
    if kind == "apply" and rng.random() < 0.3:
        n, more["caller"] = min(n, 6), True
    if kind == "apply" and rng.random() < 0.25:
        more["one_neighbour"] = True
    if kind != "apply":
        more |= dict(steps=rng.randint(10, 24), cgs2=kind == "haydock" and rng.random() < 0.25)
    return _system("", kind, n, nd, nv, nc, rng.randint(1, 4 if kind == "apply" else 3), scheme, kc, **more)


# ------------------------------------------------------------------ the state
class State:
    """A program's context and handles; freed with it."""

    def __init__(self, case):
        self.case = case
        self.ctx = bse.Context(0, torch.cuda.current_stream().cuda_stream)
        self.handles = []

    def keep(self, h):
        self.handles.append(h)
        return h

    def __del__(self):
        for h in reversed(self.handles):
            h.free()
        self.ctx.close()


def _model(c, seed):
    return synth.draw_model(1000 + seed, c["nv"], c["nc"])


def _vec(c):
    return "f64" if c["kc"] == "f64" else "f32"


def _caller_inputs(c, seed):
    """Another crystal's K_c (device), energies, dipoles and overlaps (host)."""
    g = Crystal(_model(c, seed + 500000), c["n"], c["nd"])
    return {"kc": g.kernel(), "dE": g.dE.reshape(-1).cpu().numpy(), "P": g.P.reshape(3, -1).cpu().numpy(),
            "Dv": g.Dv.cpu().numpy(), "Dc": g.Dc.cpu().numpy()}


def _handle(st, c, seed):
    caller = _caller_inputs(c, seed) if c.get("caller") else None
    co = st.keep(st.ctx.bse_build_coarse(_model(c, seed), c["n"], PREC[c["kc"]], caller["kc"].data_ptr() if caller else 0))
    scheme = SCHEME[c["scheme"]] | (bse.NB1 if c.get("one_neighbour") else 0)
    dense = {k: caller[k] for k in ("dE", "P", "Dv", "Dc")} if caller else None
    return st.keep(st.ctx.bse_interp_setup(co, c["nd"], scheme, c["width"], PREC[_vec(c)], dense))


def _network(d_in, seed):
    """He-initialised parameters in the library's flat layout."""
    r = np.random.default_rng(seed)
    dims = [d_in, WIDTH, WIDTH, WIDTH, 2]
    out = []
    for i in range(4):
        out += [r.standard_normal(dims[i + 1] * dims[i]) * math.sqrt(2.0 / dims[i]), 0.05 * r.standard_normal(dims[i + 1])]
    return np.concatenate(out).astype(np.float32)


def _vectors(c, seed):
    N = c["nv"] * c["nc"] * (c["n"] * c["nd"]) ** 3
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.randn((c["vecs"], N, 2), generator=g, device="cuda", dtype=torch.float64)
    x = torch.view_as_complex(x) / math.sqrt(2.0)
    return x if _vec(c) == "f64" else x.to(torch.complex64)


def _pair_indices(c, seed):
    """Dense points and partners closer than two coarse spacings, as the training data is sampled."""
    r = np.random.default_rng(seed)
    n, nd, L = c["n"], c["nd"], c["n"] * c["nd"]
    g = _dense_points(n, nd).numpy()
    lin = np.empty(L ** 3, dtype=np.int64)
    lin[(g[:, 0] * L + g[:, 1]) * L + g[:, 2]] = np.arange(L ** 3)
    rad = min(2 * nd, L // 2)
    offs = np.array([(a, b, e) for a in range(-rad, rad + 1) for b in range(-rad, rad + 1) for e in range(-rad, rad + 1)
                     if a * a + b * b + e * e < rad * rad])
    kd = r.integers(0, L ** 3, c["blocks"])
    h = np.mod(g[kd] - offs[r.integers(0, len(offs), c["blocks"])], L)
    return kd.astype(np.int32), lin[(h[:, 0] * L + h[:, 1]) * L + h[:, 2]].astype(np.int32)


def _batch_rows(case, seed):
    """Feature rows and targets as the training data has them."""
    t = case["bands"]
    g = torch.Generator(device="cuda").manual_seed(seed)
    X = torch.zeros((case["rows"], 6 + 2 * t), device="cuda")
    q = 0.25 * torch.randn((case["rows"], 3), generator=g, device="cuda")
    X[:, :3], X[:, 3] = q, q.norm(dim=1)
    for o in (4, 4 + t):
        X.scatter_(1, o + torch.randint(0, t, (case["rows"], 1), generator=g, device="cuda"), 1.0)
    X[:, 4 + 2 * t:] = 1.1 + 2.0 * torch.rand((case["rows"], 2), generator=g, device="cuda")
    Y = 0.4 * torch.randn((case["rows"], 2), generator=g, device="cuda")
    return X, Y


def prepare(case, seed):
    st, kind = State(case), case["kind"]
    if kind == "gradients":
        d_in = 6 + 2 * case["bands"]
        st.mlp = st.keep(st.ctx.bse_mlp_create(d_in, case["rows"], _network(d_in, seed)))
        st.X, st.Y = _batch_rows(case, seed)
    elif kind == "batch":
        st.systems, st.its = _batch_systems(case, seed), []
        for s in st.systems:
            co = st.keep(st.ctx.bse_build_coarse(s.model, s.n_coarse, bse.PREC_BF16))
            st.its.append(st.keep(st.ctx.bse_interp_setup(co, s.n_div, bse.SCHEME_M3, 1.0, bse.PREC_F32)))
        st.dirs = np.concatenate([s.pol_dirs for s in st.systems])
    elif kind == "spectrum_run":
        st.model, st.dirs = _model(case, seed), synth.POL3[:case["vecs"]].copy()
        st.omega = synth.frequency_grid(1000)
    else:
        st.it = _handle(st, case, seed)
        if kind == "apply":
            st.x = _vectors(case, seed)
            st.y = torch.empty_like(st.x)
            if case.get("learned"):
                d_in = 6 + 2 * st.it.t
                mlp = st.keep(st.ctx.bse_mlp_create(d_in, 4096, _network(d_in, seed)))
                st.ctx.bse_interp_set_learned(st.it, mlp, case["learned"])
        elif kind == "haydock":
            st.dirs = synth.POL3[:case["vecs"]].copy()
        elif kind == "pairs":
            st.kd = _pair_indices(case, seed)
            rows = case["blocks"] * st.it.t ** 2
            st.X = torch.zeros((rows, 6 + 2 * st.it.t), device="cuda")
            st.Y = torch.zeros((rows, 2), device="cuda")
    torch.cuda.synchronize()
    return st


def _batch_systems(case, seed):
    """The uneven batch's shapes (its own seeds), with models of this seed."""
    out = synth.batched_systems(case["first"], case["count"])
    for i, s in enumerate(out):
        m = s.model
        s.model = synth.draw_model(1000 * (seed + 1) + i, m.nv, m.nc, eps_inf=m.eps_inf, kappa=m.kappa)
    return out


def _flags(case):
    return bse.USE_GRAPH | (bse.REORTH_CGS2 if case.get("cgs2") else 0)


def _coefficients(a, b, pn2, steps, mixed):
    t = np.float32 if mixed else np.float64
    return {"a": a.astype(t), "b": b.astype(t), "pnorm2": pn2, "steps": steps}


def run(st):
    c, kind, ctx = st.case, st.case["kind"], st.ctx
    if kind == "apply":
        ctx.bse_apply_h(st.it, c["vecs"], st.x.data_ptr(), st.y.data_ptr())
        return st.y
    if kind == "haydock":
        a, b, pn2, steps, _ = ctx.bse_haydock_run([st.it], [c["vecs"]], st.dirs, c["steps"], _flags(c))
        return _coefficients(a, b, pn2, steps, _vec(c) == "f32")
    if kind == "batch":
        a, b, pn2, steps, _ = ctx.bse_haydock_run(st.its, [3] * len(st.its), st.dirs, c["steps"], bse.USE_GRAPH)
        return _coefficients(a, b, pn2, steps, True)
    if kind == "spectrum_run":
        co = ctx.bse_build_coarse(st.model, c["n"], PREC[c["kc"]])
        it = ctx.bse_interp_setup(co, c["nd"], SCHEME[c["scheme"]], c["width"], PREC[_vec(c)])
        a, b, pn2, steps, _ = ctx.bse_haydock_run([it], [c["vecs"]], st.dirs, c["steps"], _flags(c))
        eps = ctx.bse_spectrum(a, b, pn2, steps, synth.S_EPS / it.Nk, ETA, st.omega)
        it.free()
        co.free()
        mixed = _vec(c) == "f32"
        return _coefficients(a, b, pn2, steps, mixed) | {"eps": eps.astype(np.complex64 if mixed else np.complex128)}
    if kind == "gradients":
        g, loss = ctx.bse_mlp_gradients(st.mlp, c["rows"], st.X.data_ptr(), st.Y.data_ptr())
        return {"gradients": g, "loss": np.float32(loss)}
    ctx.bse_pairs_generate(st.it, st.kd[0], st.kd[1], st.X.data_ptr(), st.Y.data_ptr())
    return {"X": st.X, "Y": st.Y}


# ------------------------------------------------------------------- the work
def _near_offsets(nd, width):
    R2 = math.floor(width * width * nd * nd + 1e-9)
    r = int(math.floor(math.sqrt(R2)))
    return [(a, b, e) for a in range(-r, r + 1) for b in range(-r, r + 1) for e in range(-r, r + 1)
            if a * a + b * b + e * e <= R2]


def _apply_work(n, nd, nv, nc, p, scheme, kc, width=1.0, caller=False, learned=0):
    t, nk, vs = nv * nc, (n * nd) ** 3, 16 if kc == "f64" else 8
    Nc, N = t * n ** 3, t * nk
    if scheme == "m2":
        return 16.0 * N * N + 2.0 * p * N * 16, 8.0 * p * N * N
    corners = ((2 * nd - 1) / nd) ** 3 if caller else 1.0     # without the model's common basis each corner has overlaps of its own
    by = Nc * Nc * {"f64": 16, "f32": 8, "bf16": 4}[kc] + 2 * p * N * vs + N * vs / 2 + nk * corners * (nv * nv + nc * nc) * vs
    fl = 8.0 * p * Nc * Nc + 16.0 * p * N * corners * (nv + nc)
    if scheme == "m3":
        fl += 4.0 * p * N * corners * len(_near_offsets(nd, width))
    if learned:
        by += t * t * nk * 8
        fl += 8.0 * p * t * t * nk + 2 * 5.0 * p * N * math.log2(nk)
    return by, fl


def work(case):
    k = case["kind"]
    if k == "gradients":
        d = 6 + 2 * case["bands"]
        mac = d * WIDTH + 2 * WIDTH * WIDTH + 2 * WIDTH
        return {"bytes": 4.0 * (case["rows"] * (d + 2) + 2 * mac), "flops": 2.0 * case["rows"] * (3 * mac - d * WIDTH)}
    if k == "batch":
        by = fl = 0.0
        for s in synth.batched_systems(case["first"], case["count"]):
            b, f = _apply_work(s.n_coarse, s.n_div, s.model.nv, s.model.nc, 3, "m3", "bf16")
            by, fl = by + b, fl + f
        return {"bytes": by * case["steps"], "flops": fl * case["steps"]}
    c = case
    t, Nc, N = c["nv"] * c["nc"], c["nv"] * c["nc"] * c["n"] ** 3, c["nv"] * c["nc"] * (c["n"] * c["nd"]) ** 3
    if k == "pairs":
        corners = ((2 * c["nd"] - 1) / c["nd"]) ** 3
        return {"bytes": 4.0 * c["blocks"] * t * t * (8 + 2 * t), "flops": 16.0 * c["blocks"] * corners ** 2 * t * t * (c["nv"] + c["nc"])}
    by, fl = _apply_work(c["n"], c["nd"], c["nv"], c["nc"], c["vecs"], c["scheme"], c["kc"], c["width"], bool(c.get("caller")),
                         c.get("learned", 0))
    m = c.get("steps", 1)
    by, fl = by * m, fl * m
    if c.get("cgs2"):
        by, fl = by + 2 * 16.0 * c["vecs"] * N * m, fl + 16.0 * c["vecs"] * N * m * m
    if k == "spectrum_run":
        by += Nc * Nc * {"f64": 16, "f32": 8, "bf16": 4}[c["kc"]]
        fl += 8.0 * 26 * Nc * Nc / 2
    return {"bytes": by, "flops": fl}


# ------------------------------------------------- the same numbers in 64 bits
C128 = torch.complex128


def _dense_points(n, nd):
    """Integer coordinates of the dense mesh, coarse point by coarse point."""
    def cube(m):
        return torch.cartesian_prod(*[torch.arange(m)] * 3).reshape(-1, 3)
    return (cube(n)[:, None, :] * nd + cube(nd)[None, :, :]).reshape(-1, 3)


def _index(g, L):
    g = torch.remainder(g, L)
    return (g[..., 0] * L + g[..., 1]) * L + g[..., 2]


def _shape(L, kappa, head):
    """[L^3]: h or its divergent head over index differences, minimum image, half-way differences averaged."""
    d = torch.cartesian_prod(*[torch.arange(L, device="cuda", dtype=torch.float64)] * 3).reshape(-1, 3)
    near, far = torch.where(2 * d > L, d - L, d), torch.where(2 * d >= L, d - L, d)
    out = torch.zeros(L ** 3, device="cuda", dtype=torch.float64)
    for s in range(8):
        q = torch.stack([(near, far)[(s >> a) & 1][:, a] for a in range(3)], 1) / L
        if head:
            out += 1.0 / ((q * q).sum(1) + kappa ** 2)
        else:
            for G in synth.gvectors_all():
                qg = q + torch.tensor(G, device="cuda", dtype=torch.float64)
                out += math.exp(-float(G @ G)) * 4 * math.pi / ((qg * qg).sum(1) + kappa ** 2)
    return out / 8


class Crystal:
    """The model crystal on its two meshes: energies, dipoles, band gauge, overlaps, K_c."""

    def __init__(self, m, n, nd, one_neighbour=False):
        dev = lambda v: torch.tensor(np.asarray(v), device="cuda")  # noqa: E731
        self.m, self.n, self.nd, self.nv, self.nc, self.t = m, n, nd, m.nv, m.nc, m.nv * m.nc
        self.mu, self.gens = dev(m.mu), (dev(m.gen_v), dev(m.gen_c))
        self.g = _dense_points(n, nd).cuda()
        self.gc = _dense_points(n, 1).cuda()
        self.nk, self.nkc, self.ndiv = len(self.g), len(self.gc), nd ** 3
        self.Uv, self.Uc = (self._gauge(x, self.g.double() / (n * nd)) for x in self.gens)
        self.Uvc, self.Ucc = (self._gauge(x, self.gc.double() / n) for x in self.gens)
        k = self.g.double() / (n * nd)
        band = m.e_gap + m.band_width * (1 - torch.cos(2 * math.pi * k)).sum(1)
        self.dE = band[:, None, None] + dev(m.offsets)
        pi = torch.einsum("ph,hamn->pamn", self._harmonics(k).to(C128), dev(m.dip))
        self.P = torch.einsum("pmv,pamn,pnc->apvc", self.Uv, pi, self.Uc.conj())
        j = torch.remainder(self.g, nd)
        l = torch.cartesian_prod(*[torch.arange(2, device="cuda")] * 3).reshape(-1, 3)
        self.l = l
        self.corner = _index(torch.div(self.g, nd, rounding_mode="floor")[:, None, :] + l, n)
        if one_neighbour:
            self.f = ((2 * j > nd).long()[:, None, :] == l).all(-1).double()
        else:
            self.f = torch.where(l == 1, j[:, None, :].double(), nd - j[:, None, :].double()).prod(-1) / self.ndiv
        self.Dv = torch.einsum("klmn,kmv->klnv", self.Uvc[self.corner].conj(), self.Uv)
        self.Dc = torch.einsum("klmn,kmc->klnc", self.Ucc[self.corner].conj(), self.Uc)

    @staticmethod
    def _harmonics(k):
        c, s = torch.cos(2 * math.pi * k), torch.sin(2 * math.pi * k)
        return torch.stack([torch.ones_like(c[:, 0]), c[:, 0], s[:, 0], c[:, 1], s[:, 1], c[:, 2], s[:, 2]], 1)

    @classmethod
    def _gauge(cls, gen, k):
        h = cls._harmonics(k)
        w = torch.stack([h[:, 2::2], 1 - h[:, 1::2]], 2).to(C128)
        return torch.linalg.matrix_exp(1j * torch.einsum("pas,asmn->pmn", w, gen))

    def form_factors(self, Uv, Uc, k):
        mu = torch.einsum("ph,hgmn->pgmn", self._harmonics(k).to(C128), self.mu)
        return torch.einsum("pmv,pgmn,pnc->pgvc", Uv.conj(), mu, Uc).reshape(len(Uv), 26, self.t)

    def coulomb(self):
        g = synth.gvectors_nonzero()
        return torch.tensor(4 * math.pi / (g * g).sum(1), device="cuda")

    def kernel(self):
        """K_c whole, [N_c, N_c]."""
        M = self.form_factors(self.Uvc, self.Ucc, self.gc.double() / self.n).permute(0, 2, 1).reshape(-1, 26)
        K = 2 * (M.conj() * self.coulomb()) @ M.T
        ov = torch.einsum("amv,bmw->avbw", self.Uvc, self.Uvc.conj())
        oc = torch.einsum("amc,bmd->acbd", self.Ucc.conj(), self.Ucc)
        h = _shape(self.n, self.m.kappa, False)[_index(self.gc[:, None] - self.gc[None], self.n)]
        D = torch.einsum("avbw,acbd,ab->avcbwd", ov, oc, h.to(C128)).reshape(K.shape)
        return (self.m.e_k / self.nkc) * (K - D / self.m.eps_inf)

    def to_common(self, Q):
        return torch.einsum("amv,...avc,anc->...amn", self.Uvc.conj(), Q, self.Ucc)

    def apply_kernel(self, Q):
        """K_c Q without K_c: the direct term is scalar in the common basis, the exchange has rank 26."""
        M = self.form_factors(self.Uvc, self.Ucc, self.gc.double() / self.n).permute(0, 2, 1).reshape(-1, 26)
        q = Q.reshape(len(Q), -1)
        ex = 2 * torch.einsum("ig,g,jg,pj->pi", M.conj(), self.coulomb().to(C128), M, q) if len(M) <= 4096 else \
            2 * ((q @ M) * self.coulomb()) @ M.conj().T
        h = _shape(self.n, self.m.kappa, False)[_index(self.gc[:, None] - self.gc[None], self.n)].to(C128)
        d = torch.einsum("ab,pbmn->pamn", h, self.to_common(Q))
        d = torch.einsum("amv,pamn,anc->pavc", self.Uvc, d, self.Ucc.conj())
        return (self.m.e_k / self.nkc) * (ex.reshape(Q.shape) - d / self.m.eps_inf)


class Hamiltonian:
    """H of the double-grid interpolation, applied in 64 bits: diag(dE) + F K_c F^H / N_div, and Method 3's near pairs."""

    def __init__(self, g, scheme, width, caller=None):
        self.g, self.near = g, _near_offsets(g.nd, width) if scheme == "m3" else []
        self.kc, self.dE, self.Dv, self.Dc, self.P = None, g.dE, g.Dv, g.Dc, g.P
        if caller:
            dev = lambda k, *s: torch.tensor(caller[k], device="cuda").reshape(*s)  # noqa: E731
            self.kc, self.Dv, self.Dc = caller["kc"], dev("Dv", *g.Dv.shape), dev("Dc", *g.Dc.shape)
            self.dE, self.P = dev("dE", *g.dE.shape), dev("P", *g.P.shape)
        self.common = caller is None
        lin = torch.empty(g.nk, dtype=torch.long, device="cuda")
        L = g.n * g.nd
        lin[_index(g.g, L)] = torch.arange(g.nk, device="cuda")
        head = _shape(g.n, g.m.kappa, True)
        cell = torch.div(g.g, g.nd, rounding_mode="floor")
        self.steps = []
        for o in self.near:
            d = torch.tensor(o, device="cuda")
            to = lin[_index(g.g + d, L)]
            co = torch.div(g.g + d, g.nd, rounding_mode="floor") - cell
            r = co[:, None, None, :] + g.l[None, None, :, :] - g.l[None, :, None, :]        # [k, l, l', 3]
            hd = 1.0 / (sum((x / L) ** 2 for x in o) + g.m.kappa ** 2)
            wt = hd - head[_index(r, g.n)]
            if self.common:
                wt = torch.einsum("kl,klm,km->k", g.f, wt, g.f[to])
            else:
                wt = wt[:g.ndiv]                                                             # the same in every cell
            self.steps.append((to, wt))

    def __call__(self, psi):
        g = self.g
        p = len(psi)
        X = psi.reshape(p, g.nk, g.nv, g.nc)
        x = torch.einsum("klnv,pkvc,klmc,kl->pklnm", self.Dv.conj(), X, self.Dc, g.f.to(C128))
        Q = torch.zeros((p, g.nkc, g.nv, g.nc), dtype=C128, device="cuda")
        Q.index_add_(1, g.corner.reshape(-1), x.reshape(p, -1, g.nv, g.nc))
        R = (Q.reshape(p, -1) @ self.kc.T).reshape(Q.shape) if self.kc is not None else g.apply_kernel(Q)
        s = torch.einsum("klnv,pklnm,klmc,kl->pkvc", self.Dv, R[:, g.corner], self.Dc.conj(), g.f.to(C128))
        alpha = -(g.m.e_k / g.nkc) * 4 * math.pi / g.m.eps_inf
        if self.near and self.common:
            phi = torch.einsum("kmv,pkvc,knc->pkmn", g.Uv.conj(), X, g.Uc)
            u = torch.zeros_like(phi)
            for to, wt in self.steps:
                u += wt[:, None, None] * phi[:, to]
            s = s + alpha * torch.einsum("kmv,pkmn,knc->pkvc", g.Uv, u, g.Uc.conj())
        elif self.near:
            Uv, Uc = g.Uvc[g.corner], g.Ucc[g.corner]
            x = torch.einsum("klmv,pklvc,klnc->pklmn", Uv.conj(), x, Uc).reshape(p, g.nkc, g.ndiv, 8, -1)
            xf, u = x.reshape(p, g.nk, 8, -1), torch.zeros_like(x)
            for to, wt in self.steps:
                for lp in range(8):
                    u += wt[None, None, :, :, lp, None] * xf[:, to, lp].reshape(p, g.nkc, g.ndiv, 1, -1)
            u = u.reshape(p, g.nk, 8, g.nv, g.nc)
            u = torch.einsum("klmv,pklmn,klnc->pklvc", Uv, u, Uc.conj())
            s = s + alpha * torch.einsum("klnv,pklnm,klmc,kl->pkvc", self.Dv, u, self.Dc.conj(), g.f.to(C128))
        return (self.dE * X + s / g.ndiv).reshape(p, -1)

    def method2(self):
        """Method 2's H, whole."""
        g = self.g
        F = torch.zeros((g.nk, g.t, g.nkc, g.t), dtype=C128, device="cuda")
        blk = torch.einsum("klnv,klmc,kl->klvcnm", self.Dv, self.Dc.conj(), g.f.to(C128)).reshape(g.nk, 8, g.t, g.t)
        for l in range(8):
            F[torch.arange(g.nk), :, g.corner[:, l]] += blk[:, l]
        F = F.reshape(g.nk * g.t, -1)
        alpha = -(g.m.e_k / g.nkc) * 4 * math.pi / g.m.eps_inf
        ov = torch.einsum("amv,bmw->avbw", g.Uvc, g.Uvc.conj())
        oc = torch.einsum("amc,bmd->acbd", g.Ucc.conj(), g.Ucc)
        A = alpha * torch.einsum("avbw,acbd->avcbwd", ov, oc).reshape(g.nkc, g.t, g.nkc, g.t)
        hc = _shape(g.n, g.m.kappa, True)[_index(g.gc[:, None] - g.gc[None], g.n)]
        hd = _shape(g.n * g.nd, g.m.kappa, True)[_index(g.g[:, None] - g.g[None], g.n * g.nd)]
        K = g.kernel() - (A * hc[:, None, :, None]).reshape(g.nkc * g.t, -1)
        H = (F @ A.reshape(K.shape) @ F.conj().T).reshape(g.nk, g.t, g.nk, g.t) * hd[:, None, :, None]
        return (H.reshape(g.nk * g.t, -1) + F @ K @ F.conj().T) / g.ndiv + torch.diag(self.dE.reshape(-1)).to(C128)


def _recursion(H, P, m, cgs2):
    """Lanczos from each row of P: a, b, ||P||^2."""
    p = len(P)
    pn2 = (P.abs() ** 2).sum(1)
    a, b = np.zeros((p, m)), np.zeros((p, m + 1))
    psi, prev = P / pn2.sqrt()[:, None], torch.zeros_like(P)
    basis = [psi]
    for i in range(m):
        w = H(psi)
        a[:, i] = (psi.conj() * w).sum(1).real.cpu().numpy()
        w = w - torch.tensor(a[:, i], device="cuda")[:, None] * psi - torch.tensor(b[:, i], device="cuda")[:, None] * prev
        if cgs2:
            V = torch.stack(basis, 1)
            for _ in range(2):
                w = w - torch.einsum("pjk,pj->pk", V, torch.einsum("pjk,pk->pj", V.conj(), w))
        bn = (w.abs() ** 2).sum(1).sqrt()
        b[:, i + 1] = bn.cpu().numpy()
        prev, psi = psi, w / bn[:, None]
        if cgs2:
            basis.append(psi)
    return {"a": a, "b": b, "pnorm2": pn2.cpu().numpy(), "steps": None}


def _fraction(r, m, pref, omega):
    z = omega + 1j * ETA
    out = []
    for a, b, n2 in zip(r["a"], r["b"], r["pnorm2"]):
        g = 1.0 / (z - a[m - 1])
        for i in range(m - 2, -1, -1):
            g = 1.0 / (z - a[i] - b[i + 1] ** 2 * g)
        out.append(1.0 - pref * n2 * g)
    return np.array(out)


def _layers(flat, d_in):
    """The network's matrices as the library applies them (BF16 values) and its FP32 biases, in 64 bits."""
    dims, o, out = [d_in, WIDTH, WIDTH, WIDTH, 2], 0, []
    p = torch.tensor(flat, device="cuda")
    for i in range(4):
        w = p[o:o + dims[i + 1] * dims[i]].to(torch.bfloat16).double().reshape(dims[i + 1], dims[i])
        o += dims[i + 1] * dims[i]
        out.append((w.requires_grad_(), p[o:o + dims[i + 1]].double().requires_grad_()))
        o += dims[i + 1]
    return out


def _forward(layers, x):
    for i, (w, b) in enumerate(layers):
        x = x @ w.T + b
        if i < 3:
            x = torch.nn.functional.gelu(x)
    return x


def _learned_term(g, flat, radius, psi):
    """The Hermitian stencil of the network, as a periodic convolution."""
    L, t, p = g.n * g.nd, g.t, len(psi)
    offs = torch.tensor([(a, b, c) for a in range(-radius, radius + 1) for b in range(-radius, radius + 1)
                         for c in range(-radius, radius + 1) if a * a + b * b + c * c < radius * radius], device="cuda")
    avg = g.dE.reshape(g.nk, t).mean(0)
    q = offs.double() / L
    one = torch.eye(t, device="cuda", dtype=torch.float64)
    with torch.no_grad():
        layers = _layers(flat, 6 + 2 * t)
        out = []
        for qo in q:
            x = torch.cat([qo, qo.norm()[None]]).expand(t, t, 4)
            e1, e2 = one[:, None].expand(t, t, t), one[None].expand(t, t, t)
            d = torch.stack([avg[:, None].expand(t, t), avg[None].expand(t, t)], 2)
            out.append(torch.view_as_complex(_forward(layers, torch.cat([x, e1, e2, d], 2).reshape(t * t, -1)).contiguous()))
    T = torch.stack(out).reshape(-1, t, t)
    lin = {tuple(o): i for i, o in enumerate(offs.tolist())}
    neg = torch.tensor([lin[(-a, -b, -c)] for a, b, c in offs.tolist()], device="cuda")
    T = (T + T[neg].conj().transpose(1, 2)) / (2 * g.nk)
    ker = torch.zeros((t, t, L ** 3), dtype=C128, device="cuda")
    ker[:, :, _index(offs, L)] = T.permute(1, 2, 0)
    at = _index(g.g, L)
    f = torch.zeros((p, t, L ** 3), dtype=C128, device="cuda")
    f[:, :, at] = psi.reshape(p, g.nk, t).transpose(1, 2)
    F = lambda v: torch.fft.fftn(v.reshape(*v.shape[:-1], L, L, L), dim=(-3, -2, -1)).reshape(v.shape)  # noqa: E731
    f = torch.einsum("abx,pbx->pax", F(ker), F(f))
    f = torch.fft.ifftn(f.reshape(p, t, L, L, L), dim=(-3, -2, -1)).reshape(p, t, -1)
    return f[:, :, at].transpose(1, 2).reshape(p, -1)


def _exact_pairs(c, seed):
    g = Crystal(_model(c, seed), c["n"], c["nd"])
    L, t, B = c["n"] * c["nd"], g.t, c["blocks"]
    k1, k2 = (torch.tensor(v, device="cuda").long() for v in _pair_indices(c, seed))
    M = [g.form_factors(g.Uv[k], g.Uc[k], g.g[k].double() / L) for k in (k1, k2)]
    K = 2 * torch.einsum("bgi,g,bgj->bij", M[0].conj(), g.coulomb().to(C128), M[1])
    ov = torch.einsum("bmv,bmw->bvw", g.Uv[k1], g.Uv[k2].conj())
    oc = torch.einsum("bmc,bmd->bcd", g.Uc[k1].conj(), g.Uc[k2])
    h = _shape(L, g.m.kappa, False)[_index(g.g[k1] - g.g[k2], L)].to(C128)
    K = (g.m.e_k / g.nk) * (K - torch.einsum("bvw,bcd,b->bvcwd", ov, oc, h).reshape(B, t, t) / g.m.eps_inf)
    F = [torch.einsum("blnv,blmc,bl->blvcnm", g.Dv[k], g.Dc[k].conj(), g.f[k].to(C128)).reshape(B, 8, t, t) for k in (k1, k2)]
    Kc = g.kernel().reshape(g.nkc, t, g.nkc, t)
    for l in range(8):
        for lp in range(8):
            K = K - F[0][:, l] @ Kc[g.corner[k1, l], :, g.corner[k2, lp]] @ F[1][:, lp].conj().transpose(1, 2) / g.ndiv
    d = torch.remainder(g.g[k1] - g.g[k2], L)
    q = torch.where(2 * d >= L, d - L, d).double() / L
    X = torch.zeros((B, t, t, 6 + 2 * t), dtype=torch.float64, device="cuda")
    X[..., :3], X[..., 3] = q[:, None, None], q.norm(dim=1)[:, None, None]
    X[..., 4:4 + t] = torch.eye(t, device="cuda", dtype=torch.float64)[None, :, None]
    X[..., 4 + t:4 + 2 * t] = torch.eye(t, device="cuda", dtype=torch.float64)[None, None]
    dE = g.dE.reshape(g.nk, t)
    X[..., 4 + 2 * t], X[..., 5 + 2 * t] = dE[k1][:, :, None], dE[k2][:, None, :]
    return {"X": X.reshape(B * t * t, -1), "Y": torch.view_as_real((K * g.nk).contiguous()).reshape(-1, 2)}


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "gradients":
        d_in = 6 + 2 * c["bands"]
        layers = _layers(_network(d_in, seed), d_in)
        X, Y = _batch_rows(c, seed)
        loss = ((_forward(layers, X.double()) - Y.double()) ** 2).sum() / c["rows"]
        loss.backward()
        return {"gradients": torch.cat([v.grad.reshape(-1) for w in layers for v in w]), "loss": loss.detach()}
    if kind == "pairs":
        return _exact_pairs(c, seed)
    if kind == "batch":
        out = []
        for s in _batch_systems(c, seed):
            g = Crystal(s.model, s.n_coarse, s.n_div)
            H = Hamiltonian(g, "m3", 1.0)
            out.append(_recursion(H, H.P.reshape(3, -1), c["steps"], False))
        return {k: np.concatenate([o[k] for o in out]) for k in ("a", "b", "pnorm2")} | {"steps": None}
    g = Crystal(_model(c, seed), c["n"], c["nd"], bool(c.get("one_neighbour")))
    H = Hamiltonian(g, c["scheme"], c["width"], _caller_inputs(c, seed) if c.get("caller") else None)
    if kind == "apply":
        x = _vectors(c, seed).to(C128)
        y = H(x)
        if c.get("learned"):
            y = y + _learned_term(g, _network(6 + 2 * g.t, seed), c["learned"], x)
        return y
    P = H.P.reshape(3, -1)[:c["vecs"]]
    if c["scheme"] == "m2":
        dense = H.method2()
        r = _recursion(lambda v: v @ dense.T, P, c["steps"], c["cgs2"])
    else:
        r = _recursion(H, P, c["steps"], c["cgs2"])
    if kind == "spectrum_run":
        r["eps"] = _fraction(r, c["steps"], synth.S_EPS / g.nk, synth.frequency_grid(1000))
    return r
