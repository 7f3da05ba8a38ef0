"""Performance cases of the Cahn-Hilliard ensemble engine: what a user has it do.

Every case is one pass through the public entry points of `paper_1911_03386_gb300` on
inputs made from a seed.  Kinds:

  advance     an ensemble or an uneven batch of runs is advanced by `steps` time steps with
              beta sampled every `every` steps, then fields, observables and the running
              averages are read back to the host (the loop of a coarsening study: advance
              to the next snapshot, read it);
  field       a device field owned by the caller is advanced in place by
              ch_step_field_noalloc (host frameworks that own all device memory);
  serve       a burst of single-run requests is submitted to a server and awaited;
  statistics  moments, histogram and trend of a dense device array of beta series;
  droplets    Model 1 populations integrated on the device.

Starts: "noise" is the library's own start (C0 + 0.1 (2u - 1), counter-based draws);
"domains" is a field that has already separated into domains of C near +-1 with interfaces
of the equilibrium width, which is what a coarsening run holds for all but the first few
hundred of its 20 000 to 200 000 steps.
"""
import math

import numpy as np
import torch

import paper_1911_03386_gb300 as ch

TWO_PI = 2.0 * math.pi


def listed():
    return [
        # one 64^2 FP64 run sampled every step: the smallest run, launches and latency count
        dict(name="single_64_fp64", kind="advance", precision="fp64", groups="1*64x64", L=TWO_PI, gamma=0.01, dt=1e-3,
             C0="0", steps=200, every=1, start="noise"),
        # the 256-run 256^2 FP64 ensemble, two sample times
        dict(name="ensemble_256_fp64", kind="advance", precision="fp64", groups="256*256x256", L=TWO_PI, gamma=0.005,
             dt=1e-3, C0="0,0.4", steps=200, every=100, start="noise"),
        # the same ensemble in single precision, in its coarsening stage
        dict(name="ensemble_256_fp32", kind="advance", precision="fp32", groups="256*256x256", L=TWO_PI, gamma=0.005,
             dt=1e-3, C0="0,0.4", steps=300, every=100, start="domains"),
        # the uneven batch (64 x 128^2, 32 x 256^2, 8 x 512^2) in single precision
        dict(name="uneven_fp32", kind="advance", precision="fp32", groups="64*128x128,32*256x256,8*512x512", L=TWO_PI,
             gamma=0.005, dt=1e-3, C0="0,0.2,0.4", steps=200, every=100, start="domains"),
        # an uneven FP64 batch with odd, oblong and ragged grids beside powers of two
        dict(name="ragged_fp64", kind="advance", precision="fp64",
             groups="8*130x97,8*96x80,4*250x250,16*128x128,4*33x130,2*300x512,1*1000x17", L=TWO_PI, gamma=0.01, dt=5e-4,
             C0="0,0.2,0.4", steps=50, every=25, start="noise"),
        # long-time coarsening ensemble of 1024^2 runs, single precision (compensated fields)
        dict(name="long_1024_fp32", kind="advance", precision="fp32", groups="16*1024x1024", L=TWO_PI, gamma=0.0025,
             dt=5e-4, C0="0,0.3", steps=200, every=100, start="domains"),
        # the same in double precision
        dict(name="long_1024_fp64", kind="advance", precision="fp64", groups="16*1024x1024", L=TWO_PI, gamma=0.0025,
             dt=5e-4, C0="0,0.3", steps=40, every=20, start="domains"),
        # the paper's campaign at L = 4 pi (512^2, asymmetric mixture), sampled every 10 steps
        dict(name="campaign_512_fp32", kind="advance", precision="fp32", groups="64*512x512", L=2 * TWO_PI, gamma=0.01,
             dt=0.0012, C0="0.45", steps=100, every=10, start="domains"),
        # a caller-owned 512^2 device field advanced without allocation
        dict(name="field_512_noalloc", kind="field", nx=512, ny=512, L=TWO_PI, gamma=0.01, dt=1e-3, C0="0", steps=20,
             start="domains"),
        # a burst of double-precision requests of mixed size and horizon
        dict(name="serve_fp64", kind="serve", precision="fp64", sizes="64,128,256", requests=24, hmin=100, hmax=400,
             L=TWO_PI, gamma=0.005, dt=1e-3),
        # statistics of 1024 runs x 8192 sample times, some of them diverged
        dict(name="beta_statistics", kind="statistics", members=1024, samples=8192, bins=100),
        # 100 droplet populations of 512 (Model 1, the smallest of the paper's table)
        dict(name="droplets_512", kind="droplets", M=100, N=512, t_end=1e-5),
    ]


def draw(rng):
    """One more case of the ranges above (never above the largest listed work)."""
    kind = rng.choices(["even", "ragged", "field", "serve", "statistics", "droplets"], [8, 4, 2, 1, 1, 1])[0]
    if kind == "even":
        # ensembles of one size: n from 48 to 1024, powers of two, multiples of 32 and odd sizes
        n = rng.choice([64, 128, 256, 512, 1024, 32 * rng.randint(2, 24), int(round(math.exp(rng.uniform(math.log(48), math.log(900)))))])
        most = max(1, (1 << 24) // (n * n))
        m = max(1, int(round(math.exp(rng.uniform(0.0, math.log(min(256, most)))))))
        prec = rng.choice(["fp64", "fp32"])
        steps = rng.choice([10, 25, 50]) if prec == "fp64" else rng.choice([30, 75, 150])
        gamma, dt = rng.choice([(0.005, 1e-3), (0.01, 1e-3), (0.01, 0.0012), (0.0025, 5e-4)])
        start = "domains" if prec == "fp32" else rng.choice(["noise", "domains"])
        return dict(kind="advance", precision=prec, groups="%d*%dx%d" % (m, n, n), L=rng.choice([TWO_PI, 2 * TWO_PI]),
                    gamma=gamma, dt=dt, C0=rng.choice(["0", "0,0.4", "0.45", "0,0.3"]), steps=steps,
                    every=rng.choice([1, 10, steps]) if m * n * n < 1 << 20 else rng.choice([10, steps]), start=start)
    if kind == "ragged":
        gs, pts = [], 0
        for _ in range(rng.randint(2, 6)):
            nx, ny = (rng.choice([rng.randint(7, 600), 16 * rng.randint(1, 32), 1 << rng.randint(4, 9)]) for _ in range(2))
            m = rng.randint(1, 12)
            if pts + m * nx * ny <= 1 << 22:
                gs.append("%d*%dx%d" % (m, nx, ny))
                pts += m * nx * ny
        prec = rng.choice(["fp64", "fp64", "fp32"])
        return dict(kind="advance", precision=prec, groups=",".join(gs) or "2*45x77", L=TWO_PI, gamma=0.01, dt=5e-4,
                    C0=rng.choice(["0,0.2,0.4", "0.3"]), steps=rng.choice([20, 40]), every=20,
                    start="domains" if prec == "fp32" else "noise")
    if kind == "field":
        nx, ny = (rng.choice([rng.randint(40, 600), 1 << rng.randint(6, 9)]) for _ in range(2))
        return dict(kind="field", nx=nx, ny=ny, L=TWO_PI, gamma=rng.choice([0.005, 0.01]), dt=1e-3, C0="0",
                    steps=rng.randint(5, 20), start="domains")
    if kind == "serve":
        return dict(kind="serve", precision="fp64", sizes=rng.choice(["64,128", "64,128,256", "96,128,200"]),
                    requests=rng.randint(4, 24), hmin=50, hmax=rng.randint(100, 400), L=TWO_PI, gamma=0.005, dt=1e-3)
    if kind == "statistics":
        return dict(kind="statistics", members=rng.randint(32, 1024), samples=int(math.exp(rng.uniform(4, 9))),
                    bins=rng.choice([1, 50, 100, 333]))
    return dict(kind="droplets", M=rng.randint(4, 100), N=rng.choice([64, 100, 256, 512]), t_end=rng.choice([2e-6, 5e-6]))


# ---------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------
def members(case):
    """[(nx, ny, C0)] of an advance case, in order."""
    sizes = []
    for g in case["groups"].split(","):
        m, s = g.split("*")
        nx, ny = s.split("x")
        sizes += [(int(nx), int(ny))] * int(m)
    c0 = [float(x) for x in case["C0"].split(",")]
    return [(nx, ny, c0[k % len(c0)]) for k, (nx, ny) in enumerate(sizes)]


def domains(count, ny, nx, L, gamma, C0, gen):
    """count fields (count, ny, nx) in double precision on the GPU: random domains of C near
    +-1 whose interfaces have the equilibrium profile tanh(d / sqrt(2 gamma)), shares of the
    two phases for a mean near C0 (a tensor of count values)."""
    dev = "cuda"
    kx = torch.fft.rfftfreq(nx, d=1.0 / nx, device=dev, dtype=torch.float64) * (TWO_PI / L)
    ky = torch.fft.fftfreq(ny, d=1.0 / ny, device=dev, dtype=torch.float64) * (TWO_PI / L)
    k2 = ky[:, None] ** 2 + kx[None, :] ** 2
    k0 = 5.0  # wave number of the domains: a fifth of the box at L = 2 pi
    band = torch.exp(-k2 / (2.0 * k0 * k0)) * (k2 > 0)
    f = torch.randn(count, ny, nx, generator=gen, device=dev, dtype=torch.float64)
    f = torch.fft.irfft2(torch.fft.rfft2(f) * band, s=(ny, nx))
    f = f / f.std(dim=(1, 2), keepdim=True)
    # Gaussian level whose upper share is (1 + C0) / 2; rms slope k0 sqrt(2) / sqrt(2)
    f = f + math.sqrt(2.0) * torch.erfinv(C0.clamp(-0.95, 0.95))[:, None, None]
    return torch.tanh(f / (k0 * math.sqrt(2.0 * gamma)))


def domain_fields(case, mem, seed):
    """The members' start fields in order, one list of (ny, nx) device tensors."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    out, k = [], 0
    while k < len(mem):
        e = k
        while e < len(mem) and mem[e][:2] == mem[k][:2] and e - k < 64:
            e += 1
        c0 = torch.tensor([m[2] for m in mem[k:e]], device="cuda", dtype=torch.float64)
        out += list(domains(e - k, mem[k][1], mem[k][0], case["L"], case["gamma"], c0, gen))
        k = e
    return out


def noise_field(nx, ny, C0, seed, base):
    """The library's start: C0 + 0.1 (2u - 1), u = top 53 bits of SplitMix64 draw base + j nx + i."""
    g = np.uint64(0x9E3779B97F4A7C15)
    with np.errstate(over="ignore"):
        z = np.uint64(seed) + (np.arange(base, base + nx * ny, dtype=np.uint64) + np.uint64(1)) * g
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        z = z ^ (z >> np.uint64(31))
    u = (z >> np.uint64(11)).astype(np.float64) * 2.0 ** -53
    return (C0 + 0.1 * (2.0 * u - 1.0)).reshape(ny, nx)


def requests(case, seed):
    """The burst: (n, C0, stream seed, horizon) per request, the sizes in turn."""
    rng = np.random.default_rng([seed, 11])
    sizes = [int(s) for s in case["sizes"].split(",")]
    return [(sizes[k % len(sizes)], float(rng.uniform(0.0, 0.5)), int(rng.integers(1, 2 ** 62)),
             int(rng.integers(case["hmin"], case["hmax"] + 1))) for k in range(case["requests"])]


def beta_series(case, seed):
    """t (samples) and beta (members, samples) on the GPU: a common mean, a spread growing like
    sqrt(t), the last fiftieth of the runs diverged (NaN) half way."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    m, s = case["members"], case["samples"]
    t = torch.linspace(0.0, 100.0, s, device="cuda", dtype=torch.float64)
    z = torch.randn(m, s, generator=gen, device="cuda", dtype=torch.float64)
    beta = 0.28 + torch.sqrt(0.0056 * t)[None, :] * z
    bad = m // 50
    if bad:
        beta[m - bad:, s // 2:] = float("nan")
    return t, beta


def precision(case):
    return ch.CH_FP64 if case["precision"] == "fp64" else ch.CH_FP32


def prepare(case, seed):
    s = dict(case)
    if case["kind"] == "advance":
        mem = members(case)
        descs, base = [], 0
        for nx, ny, c0 in mem:
            descs.append(dict(nx=nx, ny=ny, L=case["L"], gamma=case["gamma"], dt=case["dt"], C0=c0, seed=seed,
                              counter_base=base))
            base += nx * ny
        e = ch.Ensemble.batch(descs, precision(case))
        e.set_sampling(case["every"], 0.0, 256)
        # host buffer of the snapshot, page-locked as the library advises for bulk copies
        s.update(e=e, mem=mem, host=torch.empty(base, dtype=torch.float64, pin_memory=True))
        if case["start"] == "domains":
            at = 0
            for f in domain_fields(case, mem, seed):
                s["host"][at:at + f.numel()].copy_(f.reshape(-1))
                at += f.numel()
            e.set_fields_ptr(s["host"].data_ptr())
        e.synchronize()
    elif case["kind"] == "field":
        s["C"] = domain_fields(case, [(case["nx"], case["ny"], float(case["C0"]))], seed)[0].contiguous()
    elif case["kind"] == "serve":
        s["server"] = ch.Server(256 << 20, precision(case), 256)
        s["reqs"] = requests(case, seed)
        s["fields"] = [np.empty((n, n)) for n, _, _, _ in s["reqs"]]
    elif case["kind"] == "statistics":
        s["t"], s["beta"] = beta_series(case, seed)
        s["mom"] = torch.empty(case["samples"], ch.CH_MOMENTS, device="cuda", dtype=torch.float64)
        s["hist"] = torch.empty(case["samples"], case["bins"] + 2, device="cuda", dtype=torch.int64)
        s["trend"] = torch.empty(4, device="cuda", dtype=torch.float64)
    else:
        s["R0"] = np.random.default_rng([seed, case["N"]]).random((case["M"], case["N"]))
    return s


# ---------------------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------------------
def run(s):
    if s["kind"] == "advance":
        e = s["e"]
        e.step(s["steps"])
        e.get_fields_ptr(s["host"].data_ptr())
        F, D, _ = e.observables()
        avg, count = e.beta_avg()
        out = dict(fields=s["host"], F=F, dFdt=D, beta_avg=avg, samples=count)
        if s["precision"] == "fp32":
            # the single-precision form's results at its precision
            out.update(fields=s["host"].to(torch.float32), F=F.astype(np.float32), dFdt=D.astype(np.float32),
                       beta_avg=avg.astype(np.float32))
        elif len(s["mem"]) == 1:
            out["series"] = e.series(0, 256)  # t, F, dF/dt, beta per sample of a single run
        return out
    if s["kind"] == "field":
        ch.ch_step_field_noalloc(s["C"].data_ptr(), s["nx"], s["ny"], s["L"], s["gamma"], s["dt"], s["steps"],
                                 torch.cuda.current_stream().cuda_stream)
        return s["C"]
    if s["kind"] == "serve":
        sv = s["server"]
        ids = [sv.submit(nx=n, ny=n, L=s["L"], gamma=s["gamma"], dt=s["dt"], C0=c0, seed=sd, nsteps=h, every=50,
                         field_out=f) for (n, c0, sd, h), f in zip(s["reqs"], s["fields"])]
        res = [sv.wait(i) for i in ids]
        keys = ("F", "dFdt", "beta", "beta_avg")
        return dict(results=np.array([[r[k] for k in keys] for r in res]),
                    fields=np.concatenate([f.ravel() for f in s["fields"]]))
    if s["kind"] == "statistics":
        st = torch.cuda.current_stream().cuda_stream
        m, n = s["members"], s["samples"]
        ch.ch_stats_moments(s["t"].data_ptr(), s["beta"].data_ptr(), m, n, n, s["mom"].data_ptr(), st)
        ch.ch_stats_histogram(s["beta"].data_ptr(), m, n, n, -2.0, 2.5, s["bins"], s["hist"].data_ptr(), st)
        ch.ch_stats_trend(s["mom"].data_ptr(), n, 20.0, 100.0, 20.0, 100.0, s["trend"].data_ptr(), st)
        return dict(moments=s["mom"], histogram=s["hist"], trend=s["trend"])
    R, ser, steps = ch.ch_droplets_run(s["R0"], s["t_end"], [0.0, 0.5 * s["t_end"], s["t_end"]])
    return dict(R=R, series=ser, steps=steps)


def work(case):
    """Least data moved (inputs read once, outputs written once) and operations of a pass: 33
    per grid point and step (stencil 15, row recurrences 8, column recurrences 8, update 2)."""
    if case["kind"] == "advance":
        pts = sum(nx * ny for nx, ny, _ in members(case))
        elt = 8 if case["precision"] == "fp64" else 4
        return dict(bytes=2 * elt * pts + 8 * pts, flops=33 * pts * case["steps"])  # + the snapshot
    if case["kind"] == "field":
        pts = case["nx"] * case["ny"]
        return dict(bytes=16 * pts, flops=33 * pts * case["steps"])
    if case["kind"] == "serve":
        mean = sum(int(x) ** 2 for x in case["sizes"].split(",")) / len(case["sizes"].split(","))
        pts = case["requests"] * mean
        return dict(bytes=8 * pts, flops=33 * pts * 0.5 * (case["hmin"] + case["hmax"]))
    if case["kind"] == "statistics":
        v = case["members"] * case["samples"]
        return dict(bytes=8 * v + 8 * case["samples"] * (case["bins"] + 9), flops=12 * v)
    # a droplet of radius below (3 t)^(1/3) vanishes by t, about 270 accepted and rejected steps
    # each; 250 operations per droplet and step
    gone = case["N"] * (3.0 * case["t_end"]) ** (1.0 / 3.0)
    return dict(bytes=16 * case["M"] * case["N"], flops=250 * case["M"] * case["N"] * 270 * gone)


# ---------------------------------------------------------------------------------------
# the same in plain torch, 64 bits
# ---------------------------------------------------------------------------------------
class Plain:
    """The scheme on a stack of fields (count, ny, nx) by FFT solves along rows and columns."""

    def __init__(self, nx, ny, L, gamma, dt):
        self.hx, self.hy, self.gamma, self.dt = L / nx, L / ny, gamma, dt

        def symbol(n, h):
            k = torch.arange(n // 2 + 1, device="cuda", dtype=torch.float64)
            return 1.0 + gamma * dt * (4.0 / h ** 2 * torch.sin(math.pi * k / n) ** 2) ** 2

        self.sx, self.sy = symbol(nx, self.hx), symbol(ny, self.hy)

    def lap(self, f):
        return ((torch.roll(f, -1, 2) - 2.0 * f + torch.roll(f, 1, 2)) / self.hx ** 2
                + (torch.roll(f, -1, 1) - 2.0 * f + torch.roll(f, 1, 1)) / self.hy ** 2)

    def mu(self, C):
        return C * C * C - C - self.gamma * self.lap(C)

    def step(self, C):
        R = self.dt * self.lap(self.mu(C))
        W = torch.fft.irfft(torch.fft.rfft(R, dim=2) / self.sx, n=C.shape[2], dim=2)
        return C + torch.fft.irfft(torch.fft.rfft(W, dim=1) / self.sy[:, None], n=C.shape[1], dim=1)

    def observables(self, C):
        mu = self.mu(C)

        def grad2(f):
            return ((torch.roll(f, -1, 2) - f) / self.hx) ** 2 + ((torch.roll(f, -1, 1) - f) / self.hy) ** 2

        hh = self.hx * self.hy
        F = hh * (0.25 * (C * C - 1.0) ** 2 + 0.5 * self.gamma * grad2(C)).sum((1, 2))
        return F, -hh * grad2(mu).sum((1, 2))

    def run(self, C, steps, every):
        """Field after steps steps, and (n, F, dF/dt) of every sample taken on the way."""
        samples = []
        for n in range(steps):
            if n % every == 0:
                samples.append((n, *self.observables(C)))
            C = self.step(C)
        return C, samples


def exact(case, seed):
    if case["kind"] == "advance":
        mem = members(case)
        single = len(mem) == 1 and case["precision"] == "fp64"
        fields, Fs, Ds, avgs, base, k = [], [], [], [], 0, 0
        start = domain_fields(case, mem, seed) if case["start"] == "domains" else None
        series = None
        while k < len(mem):
            e = k
            while e < len(mem) and mem[e][:2] == mem[k][:2]:
                e += 1
            nx, ny, _ = mem[k]
            p = Plain(nx, ny, case["L"], case["gamma"], case["dt"])
            if start is not None:
                C = torch.stack(start[k:e])
                start[k:e] = [None] * (e - k)
            else:
                C = torch.stack([torch.from_numpy(noise_field(nx, ny, mem[q][2], seed, base + (q - k) * nx * ny)).cuda()
                                 for q in range(k, e)])
            C, sm = p.run(C, case["steps"], case["every"])
            F, D = p.observables(C)
            b = [(-(n * case["dt"] / f) * d) for n, f, d in sm]
            fields.append(C.reshape(-1).cpu())
            Fs.append(F.cpu())
            Ds.append(D.cpu())
            avgs.append(torch.stack(b).mean(0).cpu())
            if single:
                series = torch.stack([torch.stack([torch.full_like(f, n * case["dt"]), f, d, x], 1)[0]
                                      for (n, f, d), x in zip(sm, b)]).cpu()
            base += (e - k) * nx * ny
            k = e
        out = dict(fields=torch.cat(fields), F=torch.cat(Fs), dFdt=torch.cat(Ds), beta_avg=torch.cat(avgs), samples=None)
        if single:
            out["series"] = series[-256:]
        return out
    if case["kind"] == "field":
        C = domain_fields(case, [(case["nx"], case["ny"], float(case["C0"]))], seed)[0][None]
        return Plain(case["nx"], case["ny"], case["L"], case["gamma"], case["dt"]).run(C, case["steps"], 1 << 30)[0][0]
    if case["kind"] == "serve":
        rows, fields = [], []
        for n, c0, sd, h in requests(case, seed):
            p = Plain(n, n, case["L"], case["gamma"], case["dt"])
            C, sm = p.run(torch.from_numpy(noise_field(n, n, c0, sd, 0)).cuda()[None], h, 50)
            F, D = (float(x[0]) for x in p.observables(C))
            t1 = 0.2 * h * case["dt"]
            b = [float(-(q * case["dt"] / f[0]) * d[0]) for q, f, d in sm if q * case["dt"] >= t1]
            rows.append([F, D, -(h * case["dt"] / F) * D, sum(b) / len(b) if b else float("nan")])
            fields.append(C.reshape(-1).cpu())
        return dict(results=np.array(rows), fields=torch.cat(fields))
    if case["kind"] == "statistics":
        t, beta = beta_series(case, seed)
        ok = torch.isfinite(beta)
        c = ok.sum(0).to(torch.float64)
        z = torch.where(ok, beta, torch.zeros_like(beta))
        m1 = z.sum(0) / c
        d = torch.where(ok, beta - m1, torch.zeros_like(beta))
        mom = torch.stack([t, c, m1] + [(d ** p).sum(0) / c for p in (2, 3, 4)], 1)
        return dict(moments=mom, histogram=None, trend=None)
    return None
