"""Performance cases: the calls a program that uses this synthesizer makes.

A string is stepped strictly one sample after another, so a call's time is its
steps times the time of a step, whatever the note's length: the cases render
stretches of notes (64 samples to a quarter of a second) and vary what
matters: how many strings run at once (1 to 4096), how large their grids are
(f0 from 27 Hz at 96 kHz to 2 kHz at 48 kHz, alpha 1 to 10), the excitation,
f0 modulation, the output channel, and the entry point: one string to host
memory, one string on the device, the call without device allocation, a batch
continued block by block, the note server, the dataset renderer, and forward
plus gradient.  String parameters come from ``workloads`` (the ranges of the
repository's benchmarks), except that hammers weigh up to 5 g and strike at up
to 2.5 m/s and that blocks with bowed strings are at most 1024 samples: harder
blows on low, strongly nonlinear strings and longer bowed notes amplify the
rounding of any 32-bit state a thousandfold and more within a tenth of a
second, so two sound programs part there.  Neither changes what a step costs.

``exact`` steps the same scheme in 64 bits with plain torch operations: the
transverse system by cyclic reduction, alternating with the longitudinal one
until both agree; gradients by the complex step.
"""

from __future__ import annotations

import copy
import math

import numpy as np
import torch
import torch.nn.functional as F

from paper_2311_18505_gb300 import dataset, grad, sfd
from paper_2311_18505_gb300 import workloads as W


# ------------------------------------------------------------------ the cases

def listed() -> list[dict]:
    return [
        # a real-time host asks for one audio buffer at a time: a bowed note of
        # a linear string, continued 64 samples per call into host memory
        dict(name="live_64", kind="live", alpha=1.0, samples=64),
        # an audio thread that may not allocate renders a short struck or plucked note
        dict(name="oneshot_1024", kind="oneshot", f0_lo=200.0, f0_hi=1000.0, samples=1024),
        # one linear note (110 Hz, N_t = 101), a quarter of a second on the device
        dict(name="note_linear", kind="note", f0=110.0, alpha=1.0, samples=12000),
        # the same string with alpha = 3 (the nonlinear single-string workload)
        dict(name="note_nonlinear", kind="note", f0=110.0, alpha=3.0, samples=4800),
        # 256 strings of mixed excitation (40-1000 Hz), the next block of each
        dict(name="stream_mixed_256", kind="stream", strings=256, f0_lo=40.0, f0_hi=1000.0, fs=48000.0,
             modulated=False, samples=1024),
        # 1000 strings of a polyphonic piece and an odd block length
        dict(name="stream_1000", kind="stream", strings=1000, f0_lo=40.0, f0_hi=1000.0, fs=48000.0,
             modulated=False, samples=513),
        # the 4096-string batch with vibrato or glissando (30-2000 Hz)
        dict(name="stream_modulated_4096", kind="stream", strings=4096, f0_lo=30.0, f0_hi=2000.0, fs=48000.0,
             modulated=True, samples=512),
        # bass strings at a studio rate: the largest grids (N_t 100-440, N_l up to 1700)
        dict(name="stream_bass_96k", kind="stream", strings=64, f0_lo=27.5, f0_hi=60.0, fs=96000.0,
             modulated=False, samples=1024),
        # a burst of note requests through the server, 1024-sample chunks, ragged lengths
        dict(name="server_512", kind="server", notes=512, max_samples=4096, chunk=1024),
        # dataset construction: both channels of randomised notes (vibrato,
        # glissando, bow envelopes) into host arrays
        dict(name="dataset_192", kind="dataset", items=192, samples=600),
        # parameter fitting: forward and adjoint of plucked and struck strings
        dict(name="grad_64", kind="grad", strings=64, samples=1200, bowed=False, output="transverse"),
        # ... and of bowed strings
        dict(name="grad_bow_12", kind="grad", strings=12, samples=600, bowed=True, output="transverse"),
    ]


def _log_int(rng, lo, hi) -> int:
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng) -> dict:
    kind = rng.choice(["live", "oneshot", "note", "stream", "stream", "stream", "server", "dataset", "grad"])
    if kind == "live":
        return dict(kind=kind, alpha=rng.choice([1.0, round(rng.uniform(1.5, 8.0), 3)]), samples=_log_int(rng, 64, 1024))
    if kind == "oneshot":
        lo = rng.uniform(80.0, 600.0)
        return dict(kind=kind, f0_lo=lo, f0_hi=lo * rng.uniform(1.2, 2.0), samples=_log_int(rng, 128, 2400))
    if kind == "note":
        return dict(kind=kind, f0=round(math.exp(rng.uniform(math.log(50.0), math.log(1500.0))), 3),
                    alpha=rng.choice([1.0, round(rng.uniform(1.2, 6.0), 3)]), samples=_log_int(rng, 480, 4800))
    if kind == "stream":
        if rng.random() < 0.25:
            return dict(kind=kind, strings=_log_int(rng, 8, 64), f0_lo=27.5, f0_hi=rng.uniform(35.0, 60.0), fs=96000.0,
                        modulated=False, samples=_log_int(rng, 256, 1024))
        return dict(kind=kind, strings=_log_int(rng, 32, 4096), f0_lo=rng.uniform(30.0, 200.0),
                    f0_hi=rng.uniform(500.0, 2000.0), fs=48000.0, modulated=rng.random() < 0.5,
                    samples=_log_int(rng, 256, 600))
    if kind == "server":
        return dict(kind=kind, notes=_log_int(rng, 64, 512), max_samples=_log_int(rng, 1024, 4096), chunk=1024)
    if kind == "dataset":
        return dict(kind=kind, items=_log_int(rng, 32, 192), samples=_log_int(rng, 300, 600))
    bowed = rng.random() < 0.3
    return dict(kind="grad", strings=_log_int(rng, 4, 12 if bowed else 64), samples=_log_int(rng, 240, 600 if bowed else 1200),
                bowed=bowed, output="transverse")


def _string(rng, lo=40.0, hi=1000.0, kinds=("pluck", "hammer", "bow"), fs=48000.0) -> dict:
    d = W.random_string(rng, lo, hi, kinds, fs=fs)
    if d["excitation"]["kind"] == "hammer":
        d["excitation"].update(mass=float(rng.uniform(1e-3, 5e-3)), vel=float(rng.uniform(0.5, 2.5)))
    return d


def _strings(case: dict, seed: int) -> list[dict]:
    """The strings (parameter dictionaries) of a case."""
    rng = np.random.Generator(np.random.PCG64([seed & 0x7fffffff, 17]))
    kind = case["kind"]
    if kind == "live":
        return [dict(_string(rng, 60.0, 400.0, ("bow",)), alpha=case["alpha"])]
    if kind == "oneshot":
        return [_string(rng, case["f0_lo"], case["f0_hi"], ("pluck", "hammer"))]
    if kind == "note":
        return [W.make(f0=case["f0"], alpha=case["alpha"], pickup=float(rng.uniform(0.55, 0.9)),
                       excitation={"kind": "pluck", "amp": float(rng.uniform(0.5e-3, 2e-3)),
                                   "pos": float(rng.uniform(0.1, 0.5))})]
    if kind == "stream":
        out = []
        for i in range(case["strings"]):
            d = _string(rng, case["f0_lo"], case["f0_hi"], fs=case["fs"])
            if case["modulated"] and i % 2 == 0:
                d["modulation"] = {"kind": "vibrato", "rate": float(rng.uniform(5.0, 7.0)), "depth": 20.0,
                                   "phase": float(rng.uniform(0, 2 * math.pi))}
            elif case["modulated"]:
                d["modulation"] = {"kind": "gliss", "depth": float(rng.choice([-1.0, 1.0])), "duration": 4.0}
            out.append(d)
        return out
    if kind == "server":
        out = []
        least = case["max_samples"] // 8
        for i in range(case["notes"]):   # the notes' lengths are the case's, their sound the seed's
            out.append(dict(_string(rng, kinds=("pluck", "hammer")), n_samples=least + i * 7919 % (case["max_samples"] - least + 1)))
        return out
    if kind == "dataset":
        dist = dataset.Distribution(seconds=case["samples"] / 48000.0, output="both", p_bow_envelope=0.5,
                                    hammer_mass=(1e-3, 5e-3), hammer_vel=(0.5, 2.5))
        items = [dataset.draw(dist, seed, i, 0) for i in range(case["items"])]
        return [dict(d, output=c, n_samples=case["samples"]) for d in items for c in ("transverse", "longitudinal")]
    kinds = ("bow",) if case["bowed"] else ("pluck", "hammer")
    return [dict(_string(rng, kinds=kinds), output=case["output"]) for _ in range(case["strings"])]


def _target(case: dict, seed: int) -> torch.Tensor:
    """What a fit compares with: decaying partials, a stand-in for recordings."""
    rng = np.random.Generator(np.random.PCG64([seed & 0x7fffffff, 18]))
    n, t = case["strings"], np.arange(case["samples"]) / 48000.0
    f, a = rng.uniform(60.0, 1000.0, (n, 1)), rng.uniform(0.2e-3, 1e-3, (n, 1))
    y = sum(a / p * np.exp(-3.0 * p * t) * np.sin(2 * math.pi * p * f * t) for p in (1, 2, 3))
    return torch.from_numpy(y.astype(np.float32))


# ------------------------------------------------------- prepare and run

class _State:
    """A context and what a program keeps in it; the context is destroyed with it."""

    def __init__(self, case: dict, pool: int):
        self.case = case
        self.ctx = sfd.sfd_ctx_create(torch.cuda.current_device(), None, pool)
        self.handles, self.batch, self.server, self.renderer = [], None, None, None

    def __del__(self):
        try:
            torch.cuda.synchronize()
            if self.server:
                sfd.sfd_server_destroy(self.server)
            if self.batch:
                sfd.sfd_batch_destroy(self.batch)
            for h in self.handles:
                sfd.sfd_string_destroy(h)
            if self.renderer:
                self.renderer.close()
            sfd.sfd_ctx_destroy(self.ctx)
        except Exception:
            pass


def prepare(case: dict, seed: int) -> _State:
    torch.cuda.init()
    kind, dicts = case["kind"], _strings(case, seed)
    st = _State(case, 256 << 20 if len(dicts) > 64 else 32 << 20)
    n = case.get("samples", 0)
    if kind in ("oneshot", "note", "stream"):
        st.out = torch.zeros(len(dicts), n, device="cuda")
    if kind == "live":
        st.handles = [sfd.string_from_dict(st.ctx, dicts[0])]
    elif kind == "oneshot":
        st.params, st.exc = sfd.params_from_dict(dicts[0]), sfd.excitation_from_dict(dicts[0]["excitation"])
    elif kind == "note":
        st.dict = dicts[0]
    elif kind == "stream":
        st.handles = [sfd.string_from_dict(st.ctx, d) for d in dicts]
        st.batch = sfd.sfd_batch_create(st.ctx, st.handles)
        sfd.sfd_batch_prepare(st.batch, [n] * len(dicts), st.out, np.arange(len(dicts)) * n)
    elif kind == "server":
        st.server = sfd.sfd_server_create(st.ctx, case["chunk"], 4096)
        st.requests = [sfd.request_from_dict(d, i) for i, d in enumerate(dicts)]
        st.lengths = [d["n_samples"] for d in dicts]
    elif kind == "dataset":
        st.renderer, st.dicts = dataset.GpuRenderer(torch.cuda.current_device(), 256 << 20), dicts
    else:
        st.dicts, st.target = dicts, _target(case, seed).cuda()
        st.theta = torch.tensor(grad.theta_of(dicts), dtype=torch.float32, device="cuda", requires_grad=True)
    return st


def run(st: _State):
    case, kind = st.case, st.case["kind"]
    n = case.get("samples", 0)
    if kind == "live":
        return sfd.sfd_synthesize(st.handles[0], n)
    if kind == "oneshot":
        sfd.sfd_synthesize_noalloc(torch.cuda.current_device(), None, st.params, st.exc, n, st.out)
        return st.out
    if kind == "note":
        s = sfd.string_from_dict(st.ctx, st.dict)
        try:
            sfd.sfd_synthesize(s, n, st.out)
        finally:
            sfd.sfd_string_destroy(s)
        return st.out
    if kind == "stream":
        # (a batch is launched once the one before has ended, as the README advises)
        torch.cuda.synchronize()
        sfd.sfd_batch_launch(st.batch)
        return st.out
    if kind == "server":
        for r in st.requests:
            sfd.sfd_server_submit(st.server, r)
        audio = [np.empty(m, np.float32) for m in st.lengths]
        left = len(audio)
        while left:
            for tag, first, data, last, _, _, _ in sfd.sfd_server_pump(st.server):
                audio[tag][first:first + len(data)] = data
                left -= last
        return np.concatenate(audio)
    if kind == "dataset":
        audio, status, _ = st.renderer(st.dicts)
        return {"transverse": audio[0::2], "longitudinal": audio[1::2], "status": status}
    st.theta.grad = None
    y = grad.synthesize(st.theta, st.dicts, n, st.ctx)
    loss = (y - st.target).square().mean()
    loss.backward()
    out = {name: st.theta.grad[:, i] for i, name in enumerate(grad.PARAM_NAMES)}
    return dict(out, audio=y.detach())


# ----------------------------------------------------------------- the work

def _grid(d: dict) -> tuple[int, int]:
    """(N_t, N_l) of a string, from the spacing rules."""
    k, m = 1.0 / d["fs"], d["modulation"]
    ratio = {"none": 1.0, "vibrato": 2.0 ** (abs(m.get("depth", 0.0)) / 1200.0),
             "gliss": 2.0 ** max(m.get("depth", 0.0), 0.0)}[m["kind"]]
    a, b, e = (2 * d["f0"] * ratio * k) ** 2, (d["kappa"] * k) ** 2, 2 * d["theta"] - 1
    h2 = (a + math.sqrt(a * a + 16 * e * b)) / (2 * e)
    nt = math.floor((1 / math.sqrt(h2)) * (1 + 1e-12))
    return nt, max(1, math.floor((1 / (2 * d["f0"] * ratio * d["alpha"] * k)) * (1 + 1e-12)))


def work(case: dict) -> dict:
    """Operations of one exact step of every string (24 per linear and 75 per
    nonlinear transverse row, 20 per longitudinal row, 10 per row and 30 per
    step for a force), the adjoint's as three times the forward's; bytes: every
    string's state in and out and four bytes for each sample."""
    flops = nbytes = 0.0
    for d in _strings(case, 0):
        nt, nl = _grid(d)
        linear, forced = d["alpha"] == 1.0, d["excitation"]["kind"] != "pluck"
        nz = 0 if linear else nl - 1
        n = d["n_samples"] if case["kind"] == "server" else case["samples"]
        step = (24 if linear else 75) * (nt - 1) + 20 * nz
        if forced:
            step += 30 + (0 if linear else 10 * (nt - 1))
        back = 3 if case["kind"] == "grad" else 0
        flops += step * n * (1 + back)
        nbytes += 4 * n * (1 + (1 if back else 0)) + 16 * (nt - 1 + nz)
    return {"bytes": nbytes, "flops": flops}


# ------------------------------------------------------- the same in 64 bits

class _Exact:
    """The linearly-implicit scheme for many strings at once, in float64 (or
    complex128 for the complex step), one row of every tensor per string.

    Solves each step for the accelerations: (theta + s0 + 2 s1, (1 - theta)/2 - s1)
    plus the strain terms on the transverse grid, a near-diagonal matrix on the
    longitudinal one, coupled through linear interpolation P and its adjoint.
    """

    def __init__(self, dicts, n, device, rows=None):
        S = len(dicts)
        self.n, self.dev = n, device
        f8 = dict(dtype=torch.float64, device=device)
        col = lambda v: torch.tensor(np.asarray(v, np.float64), **f8).reshape(S, 1)
        # the differentiable parameters, possibly complex: kappa, alpha, sigma0, sigma1, amplitude
        if rows is None:
            rows = [grad.params_of(d) for d in dicts]
        par = torch.tensor(np.asarray(rows), device=device)
        self.dt = par.dtype
        kappa, alpha, sig0, sig1, amp = (par[:, i:i + 1] for i in range(5))
        grids = [_grid(d) for d in dicts]
        nt, nl = (np.array([g[i] for g in grids]) for i in (0, 1))
        nz = np.where([d["alpha"] == 1.0 for d in dicts], 0, nl - 1)
        self.N, self.M = int(nt.max()) - 1, int(nz.max())
        N, M = self.N, self.M
        fs, L = np.array([d["fs"] for d in dicts]), np.array([d["length"] for d in dicts])
        k, ht, hl, th = col(1 / fs), col(1.0 / nt), col(1.0 / nl), col([d["theta"] for d in dicts])
        g2 = col([(2 * d["f0"]) ** 2 for d in dicts]) * k * k
        l = np.arange(1, N + 1)
        self.mu = torch.tensor(l[None] < nt[:, None], device=device).to(torch.float64)
        ghost = col([0.0 if d["boundary"] == 1 else 2.0 for d in dicts])
        self.edge = ghost * torch.tensor((l[None] == 1).astype(float) + (l[None] == nt[:, None] - 1), **f8)
        self.s0, self.s1, self.s1l = sig0 * k, sig1 * k / ht ** 2, sig1 * k / hl ** 2
        self.dg, self.og = th + self.s0 + 2 * self.s1, 0.5 * (1 - th) - self.s1
        phi = 0.5 * g2 * (alpha * alpha - 1)
        self.lam, self.mu2, self.laml = g2 / ht ** 2, kappa * kappa * k * k / ht ** 4, g2 * alpha * alpha / hl ** 2
        self.ca, self.cb, self.cz = phi / (2 * ht ** 4), phi / (2 * ht ** 3), phi / (2 * ht ** 2 * hl)
        self.coupled = M > 0
        if self.coupled:
            self.mz = torch.tensor(np.arange(1, M + 1)[None] <= nz[:, None], device=device).to(torch.float64)
            pos = np.minimum(l[None], nt[:, None]) * nl[:, None]   # P from exact integer positions
            left = pos // nt[:, None]
            self.pw = torch.tensor((pos - left * nt[:, None]) / nt[:, None], **f8)
            self.left = torch.tensor(np.minimum(left, M + 1), device=device)
            first = -((-np.arange(0, M + 2)[None] * nt[:, None]) // nl[:, None])   # first node of interval i
            self.first = torch.tensor(np.clip(first, 1, N + 1) - 1, device=device)
        # modulation and bow controls of every step
        j = np.arange(n + 1)
        rm, v, f, x = np.ones((n + 1, S)), np.zeros((n + 1, S)), np.zeros((n + 1, S)), np.full((n + 1, S), 0.5)
        zero, one = np.zeros(S), np.ones(S)
        ham, self.bow = np.zeros(S, bool), np.zeros(S, bool)
        Mh, hk, ha, ba, be, uh = zero.copy(), zero.copy(), one.copy(), zero.copy(), zero.copy(), zero.copy()
        for i, d in enumerate(dicts):
            m, e, t = d["modulation"], d["excitation"], j / d["fs"]
            if m["kind"] == "vibrato":
                rm[:, i] = 2.0 ** (2 * m["depth"] / 1200 * np.sin(2 * math.pi * m["rate"] * t + m["phase"]))
            elif m["kind"] == "gliss":
                rm[:, i] = 2.0 ** (2 * m["depth"] * np.minimum(t, m["duration"]) / m["duration"])
            if e["kind"] == "hammer":
                ham[i], x[:, i], Mh[i] = True, e["pos"], e["mass"] / (d["rho_a"] * L[i])
                hk[i], ha[i], uh[i] = e["omega"] ** (1 + e["alpha"]) / fs[i] ** 2, e["alpha"], 1 / (L[i] * fs[i])
            elif e["kind"] == "bow":
                env = e.get("envelope") or {}
                ctl = lambda key: np.interp(t, env["t"], env[key]) if env.get(key) is not None else np.full(n + 1, e[key])
                self.bow[i], ba[i], be[i] = True, e["a"] * L[i], e["eps"]
                v[:, i], x[:, i] = ctl("vel") / L[i], ctl("pos")
                f[:, i] = ctl("force") / (d["rho_a"] * L[i] ** 2) * (1.0 if e["release"] < 0 else t < e["release"])
        self.any_ham, self.any_bow = bool(ham.any()), bool(self.bow.any())
        node = np.clip(np.floor(x * nt[None]), 0, nt[None] - 1).astype(np.int64)
        tab = lambda a: torch.tensor(a, device=device)
        self.rm, self.f, self.node, self.w = tab(rm), tab(f), tab(node), tab(x * nt[None] - node)
        self.v = tab(v).to(self.dt)
        if rows is not None and self.dt.is_complex and self.any_bow:   # constant bow velocity = the amplitude
            self.v = torch.where(tab(self.bow)[None], (amp[:, 0] / tab(L))[None].expand(n + 1, S), self.v)
        self.k, self.ht = k, ht
        self.ham, self.isbow = tab(ham)[:, None], tab(self.bow)[:, None]
        self.Mh, self.hk, self.ha, self.ba, self.be = (col(a) for a in (Mh, hk, ha, ba, be))
        # pickup on either channel, output scale
        zch = np.array([d.get("output", "transverse") == "longitudinal" for d in dicts])
        po = np.array([d["pickup"] for d in dicts])
        for name, cells in (("o", nt), ("ol", nl)):
            nd = np.clip(np.floor(po * cells), 0, cells - 1).astype(np.int64)
            setattr(self, name + "_n", tab(np.minimum(nd, (N if name == "o" else M) + 1))[:, None])
            setattr(self, name + "_w", col(po * cells - nd))
        self.zch, self.L = tab(zch)[:, None], col(L)
        # initial state: the pluck triangle or the hammer at rest position
        xp = np.array([d["excitation"]["pos"] if d["excitation"]["kind"] == "pluck" else 0.5 for d in dicts])[:, None]
        xl = l[None] / nt[:, None]
        tri = np.where(xl <= xp, xl / xp, (1 - xl) / (1 - xp)) * np.array(
            [d["excitation"]["kind"] == "pluck" for d in dicts])[:, None] / L[:, None]
        self.u = (tab(tri) * amp * self.mu).to(self.dt)
        self.D = torch.zeros_like(self.u)
        self.z, self.Dz, self.az, self.xz = (torch.zeros(S, M, dtype=self.dt, device=device) for _ in range(4))
        self.uh = (col(uh) * amp).to(self.dt)
        self.Dh = self.uh.clone()
        self.y = torch.zeros(n, S, dtype=self.dt, device=device)
        self.step_no = torch.ones(1, dtype=torch.long, device=device)   # time level of the state
        self.levels = max(1, math.ceil(math.log2(N + 1)))
        self.sweeps = 6 if self.coupled else 1

    def _at(self, x, node, w):
        """Linear interpolation of nodal values (rows: nodes 1, 2, ...; ends zero)."""
        p = F.pad(x, (1, 2))
        return (1 - w) * p.gather(1, node) + w * p.gather(1, node + 1)

    def _pickup(self):
        a = self._at(self.u, self.o_n, self.o_w)
        if self.coupled:
            a = torch.where(self.zch, self._at(self.z, self.ol_n, self.ol_w), a)
        else:
            a = torch.where(self.zch, torch.zeros_like(a), a)
        return (a * self.L)[:, 0]

    def _to_t(self, z):
        p = F.pad(z, (1, 2))
        return ((1 - self.pw) * p.gather(1, self.left) + self.pw * p.gather(1, self.left + 1)) * self.mu

    def _to_l(self, f):
        """P^T f: sums of (1 - w) f and w f over the nodes of each longitudinal interval."""
        s = []
        for q in ((1 - self.pw) * f, self.pw * f):
            c = F.pad(q.cumsum(1), (1, 0)).gather(1, self.first)
            s.append(c[:, 1:] - c[:, :-1])
        return (s[0][:, 1:] + s[1][:, :-1]) * self.mz

    def _factor(self, a, b, c):
        """Cyclic reduction of the rows a x[l-1] + b x[l] + c x[l+1]."""
        ks = []
        for i in range(self.levels):
            s = 1 << i
            up = lambda v, fill: F.pad(v, (s, 0), value=fill)[:, :self.N] if s < self.N else torch.full_like(v, fill)
            dn = lambda v, fill: F.pad(v, (0, s), value=fill)[:, -self.N:] if s < self.N else torch.full_like(v, fill)
            k1, k2 = a / up(b, 1.0), c / dn(b, 1.0)
            b = b - k1 * up(c, 0.0) - k2 * dn(a, 0.0)
            a, c = -k1 * up(a, 0.0), -k2 * dn(c, 0.0)
            ks.append((s, k1[None], k2[None]))
        return ks, (1 / b)[None]

    def _solve(self, fac, d):
        ks, binv = fac
        for s, k1, k2 in ks:
            p = F.pad(d, (s, s))
            d = d - k1 * p[..., :self.N] - k2 * p[..., 2 * s:]
        return d * binv

    def _diff(self, g, x):
        """d_+[g d_- x] on nodes 1..N; g on intervals 1..N+1."""
        p = F.pad(x, (1, 1))
        q = g * (p[..., 1:] - p[..., :-1])
        return (q[..., 1:] - q[..., :-1]) * self.mu

    def step(self):
        n = self.step_no
        rm = self.rm.index_select(0, n).t()
        node, w = self.node.index_select(0, n).t(), self.w.index_select(0, n).t()
        lam, laml, ca, cb, cz = (c * rm for c in (self.lam, self.laml, self.ca, self.cb, self.cz))
        u, D, mu = self.u, self.D, self.mu
        up = F.pad(u, (1, 1))
        real = F.pad(mu, (1, 0))   # interval i touches node i - 1 or i
        g = (up[:, 1:] - up[:, :-1]) * torch.maximum(real, F.pad(mu, (0, 1)))
        dd = lambda x: F.pad(x, (0, 1))[:, 1:] - 2 * x + F.pad(x, (1, 0))[:, :-1]
        d2 = dd(u) * mu
        # at a fixed end the second difference is u_1 + u_{-1}, u_{-1} = u_1 (clamped) or -u_1
        d4 = dd(d2) + self.edge * u
        ra = lam * d2 - self.mu2 * d4 - 2 * self.s0 * D + 2 * self.s1 * dd(D)
        y3 = 2 * ca * g * g * g
        if self.coupled:
            zt = F.pad(self._to_t(self.z), (1, 1))
            y3 = y3 + 4 * cb * g * (zt[:, 1:] - zt[:, :-1])
        ra = (ra + y3[:, 1:] - y3[:, :-1]) * mu
        g2 = ca * g * g
        # interior couplings only: rows at the ends have no neighbour beyond
        inner = F.pad(mu, (1, 0))[:, :-1] * mu
        a = (self.og - g2[:, :-1]) * inner
        c = (self.og - g2[:, 1:]) * F.pad(mu, (0, 1))[:, 1:] * mu
        b = (self.dg + g2[:, :-1] + g2[:, 1:]) * mu + (1 - mu)
        fac = self._factor(a, b, c)
        J = torch.zeros_like(F.pad(u, (1, 2))).scatter(1, node, ((1 - w) / self.ht).to(self.dt))
        J = (J.scatter_add(1, node + 1, (w / self.ht).to(self.dt)))[:, 1:self.N + 1] * mu
        rhs = torch.stack([ra, J])
        if not self.coupled:
            acc, X = self._solve(fac, rhs)
            az = xz = None
        else:
            ddz = lambda x: F.pad(x, (0, 1))[:, 1:] - 2 * x + F.pad(x, (1, 0))[:, :-1]
            q = g * g
            rz = (laml * ddz(self.z) - 2 * self.s0 * self.Dz + 2 * self.s1l * ddz(self.Dz)
                  + 2 * cz * self._to_l((q[:, 1:] - q[:, :-1]) * mu)) * self.mz
            zd = 1 / (1 + self.s0 + 2 * self.s1l)
            az, xz = self.az, self.xz
            side = lambda x: F.pad(x, (0, 1))[:, 1:] + F.pad(x, (1, 0))[:, :-1]
            for _ in range(self.sweeps):
                back = torch.stack([self._diff(g, self._to_t(az)), self._diff(g, self._to_t(xz))])
                acc, X = self._solve(fac, rhs + cb * back)
                az = (rz + cz * self._to_l(self._diff(g, acc)) + self.s1l * side(az)) * zd * self.mz
                xz = (cz * self._to_l(self._diff(g, X)) + self.s1l * side(xz)) * zd * self.mz
        real_of = lambda x: x.real if x.is_complex() else x
        s = torch.zeros_like(self.uh)
        if self.any_ham:
            eta = self.uh - self._at(u, node, w)
            on = (real_of(eta) > 0) & self.ham
            G = torch.where(on, self.hk * torch.where(on, eta, torch.ones_like(eta)) ** (self.ha - 1), torch.zeros_like(eta))
            cm = 0.5 * self.Mh * G
            sh = cm * (2 * eta - self._at(acc, node, w)) / (1 + 0.5 * G + cm * self._at(X, node, w))
            s = torch.where(on, sh, s)
            self.Dh.copy_(self.Dh - torch.where(on, sh / torch.where(on, self.Mh, torch.ones_like(self.Mh)), torch.zeros_like(sh)))
            self.uh.copy_(self.uh + self.Dh)
        if self.any_bow:
            f = self.f.index_select(0, n).t()
            bv = (self._at(acc, node, w) + 2 * self._at(D, node, w)) / (2 * self.k) - self.v.index_select(0, n).t()
            cc = 0.5 * self.k * f * self._at(X, node, w)
            sg = torch.where(real_of(bv) < 0, -1.0, 1.0)
            B = bv * sg
            v, ce = B, cc * (1 - self.be)
            for _ in range(30):   # Newton from the right of the root of a convex function
                e = torch.exp(-self.ba * v)
                slope = 1 - ce * self.ba * e
                ok = real_of(slope) > 0
                v = torch.where(ok, v - (v + cc * self.be + ce * e - B) / torch.where(ok, slope, torch.ones_like(slope)), v)
            stick = real_of(B) <= real_of(cc)
            none = (f <= 0) | ~self.isbow
            ph = torch.where(stick, bv / torch.where(none, torch.ones_like(cc), cc),
                             sg * (self.be + (1 - self.be) * torch.exp(-self.ba * v)))
            s = torch.where(none, s, -self.k * self.k * f * ph)
        acc = acc + s * X
        self.D.copy_((D + acc) * mu)
        self.u.copy_(u + self.D)
        if self.coupled:
            self.az.copy_(az + s * xz)
            self.xz.copy_(xz)
            self.Dz.copy_(self.Dz + self.az)
            self.z.copy_(self.z + self.Dz)
        self.step_no += 1
        self.y.index_copy_(0, self.step_no, self._pickup()[None])

    def samples(self) -> torch.Tensor:
        """Output samples [S, n]: the two initial levels, then one per step."""
        state = [self.u, self.D, self.z, self.Dz, self.az, self.xz, self.uh, self.Dh, self.step_no]
        self.y[:2] = self._pickup()[None]
        steps = self.n - 2
        if self.dev.type == "cuda" and steps > 8:
            keep = [t.clone() for t in state]
            side = torch.cuda.Stream()
            side.wait_stream(torch.cuda.current_stream())
            with torch.cuda.stream(side):
                self.step()
            torch.cuda.current_stream().wait_stream(side)
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph):
                self.step()
            for t, v in zip(state, keep):
                t.copy_(v)
            for _ in range(steps):
                graph.replay()
        else:
            for _ in range(steps):
                self.step()
        return self.y.t()


def _samples(dicts, n, dev) -> torch.Tensor:
    """Samples of many strings, those of similar grids together."""
    if len(dicts) <= 64:
        return _Exact(dicts, n, dev).samples()
    order = np.argsort([sum(_grid(d)) for d in dicts], kind="stable")
    y = torch.empty(len(dicts), n, dtype=torch.float64, device=dev)
    for part in np.split(order, [len(order) // 2, len(order) * 7 // 8]):
        y[torch.tensor(part, device=dev)] = _Exact([dicts[i] for i in part], n, dev).samples()
    return y


def exact(case: dict, seed: int):
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    kind, dicts = case["kind"], _strings(case, seed)
    if kind == "server":
        y = _samples(dicts, max(d["n_samples"] for d in dicts), dev)
        return torch.cat([y[i, :d["n_samples"]] for i, d in enumerate(dicts)])
    if kind != "grad":
        y = _samples(dicts, case["samples"], dev)
        if kind == "dataset":
            return {"transverse": y[0::2], "longitudinal": y[1::2], "status": None}
        return y[0] if kind == "live" else y
    # theta is float32; every parameter in turn takes an imaginary step
    theta = np.asarray(grad.theta_of(dicts), np.float32).astype(np.float64)
    h, rows, many = 1e-30, [], []
    for i in range(5):
        p = theta.astype(np.complex128)
        p[:, i] += 1j * h
        rows.append(p)
        many += [grad.with_params(copy.deepcopy(d), r) for d, r in zip(dicts, theta)]
    y = _Exact(many, case["samples"], dev, np.concatenate(rows)).samples().reshape(5, len(dicts), -1)
    dy = 2 * (y[0].real - _target(case, seed).to(dev).double()) / y[0].numel()
    out = {name: (y[i].imag / h * dy).sum(1) for i, name in enumerate(grad.PARAM_NAMES)}
    return dict(out, audio=y[0].real.contiguous())
