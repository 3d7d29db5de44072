"""Performance cases of the GridSPT library: what is timed, on which inputs,
and what the results are in plain FP64.

Each case is one call (or the calls of one step) that a program makes through
the public binding. Kinds:

  orders     run_orders of one plan: the recursion delta_1 .. delta_n_max
  mixed      one graph launch of the recursion of plans of several grid sizes
  linear     make_linear_field: seeds in, delta_1(k) of every realisation out
  power      the binned P-terms of one realisation's orders
  bispectrum tree-level (or one-loop) equilateral bispectrum
  transform  c2r of a half spectrum and r2c of a real field
  train      one training step of the P-term emulator's network
  predict    the network's forward pass on a batch of parameter points
"""
import math

import numpy as np
import torch

from paper_1807_04215_gb300 import gridspt as g

COSMO = dict(omega_m=0.3, h=0.7, n_s=0.96, sigma8=0.8, gamma=0.0)
TERMS = [(1, 1), (1, 3), (2, 2), (1, 5), (2, 4), (3, 3)]


def orders(name, n, n_max, box, **opts):
    return dict(name=name, kind="orders", n=n, n_max=n_max, box=box, batch=1, form="nine_term", truncate=False,
                cut_nl=0.0, tuned=False) | opts


def listed():
    return [
        # plain GridSPT at the smallest workload: third order on 64^3 (launches count)
        orders("orders_64", 64, 3, 500.0),
        # fifth order on a 3 * 2^a grid, the middle size of the uneven batch
        orders("orders_192", 192, 5, 750.0),
        # fifth order at 256^3, the grid of the emulator's training set and of the cutoff scans
        orders("orders_256", 256, 5, 1000.0),
        # the headline: fifth order at 512^3, set up as a throughput run does (tile variants autotuned)
        orders("orders_512", 512, 5, 2000.0, tuned=True),
        # the divergence-form option (in-band results only are wanted) on a 3 * 2^a grid
        orders("divergence_384", 384, 4, 1500.0, form="divergence"),
        # the uneven batch: 128^3, 192^3 and 256^3, several seeds each, as one graph launch
        dict(name="mixed_graph", kind="mixed", n0=128, n1=192, n2=256, n_max=5, cell=3.90625, batch=2),
        # initial fields of a throughput batch, from seeds
        dict(name="linear_512", kind="linear", n=512, n_max=5, box=2000.0, batch=4),
        # the six P-terms of one 512^3 realisation in 32 log bins over 0.01-0.4 h/Mpc
        dict(name="power_512", kind="power", n=512, box=2000.0, nbins=32, k_lo=0.01, k_hi=0.4),
        # tree-level bispectrum of one 256^3 realisation in 16 shells below the linear cut
        dict(name="bispectrum_256", kind="bispectrum", n=256, box=1000.0, nbins=16, top=1.0 / 6.0, one_loop=False),
        # one large field to real space and one back: 1024^3
        dict(name="transform_1024", kind="transform", n=1024, box=4000.0, count=1),
        # one step of the emulator's training: 256 points, 3 -> 128 -> 128 -> 160, bf16 weights
        dict(name="train_step", kind="train", rows=256, n_in=3, hidden=128, out=160, bf16=True),
        # emulated P-terms of a chain of parameter points
        dict(name="predict_4096", kind="predict", rows=4096, n_in=3, hidden=128, out=160, bf16=True),
    ]


def draw(rng):
    kind = rng.choice(["orders"] * 5 + ["mixed", "linear", "power", "power", "bispectrum", "transform", "train",
                                        "predict"])
    cell = round(rng.uniform(2.0, 8.0), 4)
    if kind == "orders":
        n = rng.choice([32, 48, 64, 96, 128, 192, 256, 256, 384, 512])
        form = rng.choice(["nine_term", "nine_term", "nine_term", "divergence"])
        cut = rng.choice([0.0, 0.0, 0.0, 1.3]) if form == "nine_term" else 0.0
        return dict(kind=kind, n=n, n_max=rng.randint(2, 5), box=cell * n, batch=rng.choice([1, 2, 3]) if n < 256 else 1,
                    form=form, truncate=form == "nine_term" and rng.random() < 0.25, cut_nl=cut,
                    tuned=rng.random() < 0.25)
    if kind == "mixed":
        a, b, c = sorted(rng.sample([32, 48, 64, 96, 128, 192, 256], 3))
        return dict(kind=kind, n0=a, n1=b, n2=c, n_max=rng.randint(3, 5), cell=cell, batch=rng.randint(1, 2))
    if kind == "linear":
        n = rng.choice([64, 96, 128, 192, 256, 384, 512])
        return dict(kind=kind, n=n, n_max=rng.randint(2, 5), box=cell * n, batch=rng.randint(1, 4))
    if kind == "power":
        n = rng.choice([64, 96, 128, 192, 256, 384, 512])
        kny = math.pi / cell
        return dict(kind=kind, n=n, box=cell * n, nbins=rng.randint(1, 64), k_lo=round(kny * rng.uniform(2.0, 4.0) / n, 6),
                    k_hi=round(kny * rng.uniform(0.2, 0.99), 6))
    if kind == "bispectrum":
        n = rng.choice([32, 48, 64, 96, 128, 192, 256])
        return dict(kind=kind, n=n, box=cell * n, nbins=rng.randint(3, 16), top=round(rng.uniform(0.12, 0.33), 4),
                    one_loop=rng.random() < 0.5)
    if kind == "transform":
        n = rng.choice([32, 48, 64, 96, 128, 192, 256, 384, 512, 768])
        return dict(kind=kind, n=n, box=cell * n, count=rng.randint(1, 3))
    rows = max(1, round(2.0 ** rng.uniform(0.0, 12.0)))
    return dict(kind=kind, rows=rows, n_in=rng.randint(2, 5), hidden=rng.choice([64, 97, 128, 160, 256]),
                out=rng.randint(20, 200), bf16=rng.random() < 0.7)


# ------------------------------------------------------------------ inputs
def signed(n):
    s = torch.arange(n, device="cuda")
    return torch.where(s < n // 2, s, s - n)


def s2_grid(n):
    s = signed(n).to(torch.int32)
    z = torch.arange(n // 2, device="cuda", dtype=torch.int32)
    return (s * s)[:, None, None] + (s * s)[None, :, None] + (z * z)[None, None, :]


def linear_pk(k, c=COSMO):
    """k^n_s T_BBKS(k / Gamma)^2, normalised to sigma_8 at R = 8 Mpc/h (k: FP64 array)."""
    gam = c["gamma"] if c["gamma"] > 0 else c["omega_m"] * c["h"]

    def unit(k):
        q = np.where(k > 0, k, 1.0) / gam
        poly = 1.0 + 3.89 * q + (16.1 * q) ** 2 + (5.46 * q) ** 3 + (6.71 * q) ** 4
        t = np.log1p(2.34 * q) / (2.34 * q) * poly ** -0.25
        return np.where(k > 0, k, 1.0) ** c["n_s"] * t * t * (k > 0)

    m = 1 << 16
    lnk = np.linspace(math.log(1e-5), math.log(1e3), m + 1)
    kk = np.exp(lnk)
    x = 8.0 * kk
    w = np.where(x < 1e-3, 1.0 - x * x / 10.0, 3.0 * (np.sin(x) - x * np.cos(x)) / x ** 3)
    wt = np.ones(m + 1)
    wt[1:-1:2], wt[2:-1:2] = 4.0, 2.0
    var = (lnk[1] - lnk[0]) / 3.0 * np.dot(wt, kk ** 3 * unit(kk) * w * w) / (2.0 * math.pi ** 2)
    return c["sigma8"] ** 2 / var * unit(k)


def random_spectrum(n, box, cut, gen, amp=1.0):
    """A Gaussian half spectrum (complex64 [n][n][n/2]) with the linear spectrum
    times amp^2, Nyquist modes and |s| > cut (if any) zero."""
    f = torch.fft.rfftn(torch.randn(n, n, n, generator=gen, device="cuda"), norm="forward")[:, :, : n // 2].contiguous()
    f[n // 2] = 0
    f[:, n // 2] = 0
    s2 = s2_grid(n)
    top = 3 * (n // 2) ** 2
    pk = np.sqrt(linear_pk(2.0 * math.pi / box * np.sqrt(np.arange(top + 1, dtype=np.float64))) / box ** 3)
    if cut:
        pk[np.arange(top + 1) > cut * cut] = 0.0
    w = torch.from_numpy((amp * n ** 1.5 * pk).astype(np.float32)).cuda()
    return f * w[s2.long()]


def generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def delta1(n, n_max, box, batch, seed):
    gen = generator(seed)
    return torch.stack([random_spectrum(n, box, n / (n_max + 1), gen) for _ in range(batch)])


def buffers(plan, n_max, batch):
    spectra = torch.empty(plan.half_shape(batch, n_max - 1, 2), dtype=torch.complex64, device="cuda")
    return spectra, torch.empty(max(plan.workspace_size(), 16), dtype=torch.uint8, device="cuda")


def plan_of(c):
    kc = g.default_kcut(c["n"], c["n_max"], c["box"])
    return g.Plan(c["n"], c["n_max"], c["box"], batch=c["batch"], kcut_nl=c["cut_nl"] * kc, form=c["form"],
                  truncate=c["truncate"])


def field_set(c, seed, count):
    """delta_1 .. delta_count of one realisation, as power and bispectrum read them."""
    gen = generator(seed)
    return [random_spectrum(c["n"], c["box"], c["n"] / 6 if i == 0 else None, gen, 1.0 / (i + 1)) for i in range(count)]


def edges_of(c):
    if c["kind"] == "power":
        return [c["k_lo"] * (c["k_hi"] / c["k_lo"]) ** (i / c["nbins"]) for i in range(c["nbins"] + 1)]
    top = 2.0 * math.pi / c["box"] * c["n"] * c["top"]
    return [top * i / c["nbins"] for i in range(c["nbins"] + 1)]


def net_inputs(c, seed):
    gen = generator(seed)
    x = torch.rand(c["rows"], c["n_in"], generator=gen, device="cuda") * 2 - 1
    t = torch.randn(c["rows"], c["out"], generator=gen, device="cuda")
    mask = (torch.rand(c["out"], generator=gen, device="cuda") < 0.9).float().expand(c["rows"], -1).contiguous()
    mask[:, 0] = 1.0
    return x, t, mask, gen


def net_state(c, gen, n):
    """Parameters and Adam moments of a run in progress (step 100)."""
    m = 1e-3 * torch.randn(n, generator=gen, device="cuda")
    v = 1e-6 * (0.5 + torch.rand(n, generator=gen, device="cuda"))
    return m, v


def prepare(c, seed):
    kind = c["kind"]
    if kind == "orders":
        plan = plan_of(c)
        d1 = delta1(c["n"], c["n_max"], c["box"], c["batch"], seed)
        spectra, ws = buffers(plan, c["n_max"], c["batch"])
        if c["tuned"]:
            need = 29 * 4 * c["n"] ** 3
            g.autotune(plan, scratch=ws if ws.numel() >= need else None)
        return dict(kind=kind, plan=plan, d1=d1, spectra=spectra, ws=ws)
    if kind == "mixed":
        plans, d1s, sp, wss = [], [], [], []
        for i in range(3):
            n = c["n%d" % i]
            plans.append(g.Plan(n, c["n_max"], c["cell"] * n, batch=c["batch"]))
            d1s.append(delta1(n, c["n_max"], c["cell"] * n, c["batch"], seed * 3 + i))
            s, w = buffers(plans[-1], c["n_max"], c["batch"])
            sp.append(s)
            wss.append(w)
        return dict(kind=kind, graph=g.Batch(plans, d1s, spectra=sp, wss=wss))
    if kind == "linear":
        plan = g.Plan(c["n"], c["n_max"], c["box"], batch=c["batch"])
        out = torch.empty(plan.half_shape(c["batch"]), dtype=torch.complex64, device="cuda")
        return dict(kind=kind, plan=plan, seeds=[int(seed) * 16 + i for i in range(c["batch"])], out=out)
    if kind == "power":
        plan = g.Plan(c["n"], 5, c["box"])
        return dict(kind=kind, plan=plan, d=field_set(c, seed, 5), edges=edges_of(c),
                    ws=torch.empty(g.power_workspace_size(plan, c["nbins"]), dtype=torch.uint8, device="cuda"),
                    out=torch.empty(len(TERMS), c["nbins"], dtype=torch.float64, device="cuda"),
                    nk=torch.empty(c["nbins"], dtype=torch.int64, device="cuda"))
    if kind == "bispectrum":
        plan = g.Plan(c["n"], 5, c["box"])
        return dict(kind=kind, plan=plan, d=field_set(c, seed, 4 if c["one_loop"] else 2), edges=edges_of(c),
                    one_loop=c["one_loop"],
                    ws=torch.empty(g.bispectrum_workspace_size(plan, c["nbins"]), dtype=torch.uint8, device="cuda"))
    if kind == "transform":
        plan = g.Plan(c["n"], 2, c["box"])
        gen = generator(seed)
        spec = torch.stack([random_spectrum(c["n"], c["box"], None, gen) for _ in range(c["count"])])
        field = torch.randn(c["count"], c["n"], c["n"], c["n"], generator=gen, device="cuda")
        return dict(kind=kind, plan=plan, spec=spec, field=field, out_x=torch.empty_like(field),
                    out_k=torch.empty_like(spec))
    net = g.MLP(c["n_in"], c["hidden"], c["out"], bf16=c["bf16"], seed=int(seed) % (1 << 31))
    x, t, mask, gen = net_inputs(c, seed)
    y = torch.empty(c["rows"], c["out"], device="cuda")
    if kind == "predict":
        return dict(kind=kind, net=net, x=x, y=y)
    m, v = net_state(c, gen, net.n)
    net.m.copy_(m)
    net.v.copy_(v)
    net.step.fill_(100)
    return dict(kind=kind, net=net, x=x, t=t, mask=mask, y=y, dy=torch.empty_like(y),
                act=torch.empty(c["rows"], 4 * c["hidden"], device="cuda"), loss=torch.zeros(1, device="cuda"),
                ws=torch.empty(net.ws_bytes(c["rows"]), dtype=torch.uint8, device="cuda"))


# ------------------------------------------------------------------- calls
def run(s):
    kind = s["kind"]
    if kind == "orders":
        return g.run_orders(s["plan"], s["d1"], spectra=s["spectra"], ws=s["ws"])
    if kind == "mixed":
        return s["graph"].launch()
    if kind == "linear":
        return g.make_linear_field(s["plan"], s["seeds"], COSMO, out=s["out"])
    if kind == "power":
        for t, (i, j) in enumerate(TERMS):
            g.power(s["plan"], s["d"][i - 1], s["d"][j - 1], s["edges"], ws=s["ws"], out=s["out"][t], nk=s["nk"])
        return s["out"], s["nk"]
    if kind == "bispectrum":
        d = s["d"]
        if s["one_loop"]:
            return g.bispectrum_one_loop(s["plan"], d[0], d[1], d[2], d[3], s["edges"], ws=s["ws"])
        return g.bispectrum(s["plan"], d[0], d[1], s["edges"], ws=s["ws"])
    if kind == "transform":
        return g.c2r(s["plan"], s["spec"], out=s["out_x"]), g.r2c(s["plan"], s["field"], out=s["out_k"])
    net = s["net"]
    if kind == "predict":
        return net.forward(s["x"], y=s["y"])
    net.forward(s["x"], y=s["y"], act=s["act"])
    net.mse(s["y"], s["t"], s["mask"], s["dy"], s["loss"])
    net.backward(s["x"], s["act"], s["dy"], s["ws"])
    net.adam(1e-3)
    return dict(y=s["y"], loss=s["loss"], grad=net.grad, master=net.master, m=net.m, v=net.v, lowp=net.lowp)


# -------------------------------------------------------------------- work
def orders_work(n, n_max, batch, form):
    """Fields in and out once; the transforms and products the sources need:
    per order below n_max its real derived fields, per order formed its sources."""
    cells = float(n) ** 3
    fft = 2.5 * cells * math.log2(cells)
    f = 0.0
    for m in range(1, n_max):
        f += fft * (4 if form == "divergence" else 13 if m == 1 else 17)
    for m in range(2, n_max + 1):
        if form == "divergence":
            f += 4 * fft + 14.0 * cells * ((m + 1) // 2)
        else:
            f += 2 * fft + 44.0 * cells * ((m + 1) // 2)
    return 4.0 * cells * batch * (1 + 2 * (n_max - 1)), f * batch


def work(c):
    kind = c["kind"]
    if kind == "orders":
        b, f = orders_work(c["n"], c["n_max"], c["batch"], c["form"])
        return {"bytes": b, "flops": f}
    if kind == "mixed":
        w = [orders_work(c["n%d" % i], c["n_max"], c["batch"], "nine_term") for i in range(3)]
        return {"bytes": sum(x[0] for x in w), "flops": sum(x[1] for x in w)}
    if kind == "linear":
        modes = 2.0 / 3.0 * math.pi * (c["n"] / (c["n_max"] + 1)) ** 3
        return {"bytes": 4.0 * c["n"] ** 3 * c["batch"], "flops": 100.0 * modes * c["batch"]}
    if kind == "power":
        modes = 2.0 / 3.0 * math.pi * (c["k_hi"] * c["box"] / (2.0 * math.pi)) ** 3
        return {"bytes": 8.0 * modes * 5, "flops": 5.0 * modes * len(TERMS)}
    if kind == "bispectrum":
        r = c["n"] * c["top"]
        modes = 2.0 / 3.0 * math.pi * r ** 3
        fields, sums = (4, 3) if c["one_loop"] else (2, 1)
        f = 0.0
        for i in range(1, c["nbins"] + 1):   # a shell of radius ri needs a grid of 3 ri points a side
            pts = (3.0 * r * i / c["nbins"] + 1.0) ** 3
            f += (fields + 1) * 2.5 * pts * math.log2(max(pts, 2.0)) + 6.0 * sums * pts
        return {"bytes": 8.0 * modes * fields, "flops": f}
    if kind == "transform":
        cells = float(c["n"]) ** 3 * c["count"]
        return {"bytes": 16.0 * cells, "flops": 5.0 * cells * 3 * math.log2(c["n"])}
    i, h, o, r = c["n_in"], c["hidden"], c["out"], c["rows"]
    params = i * h + h + h * h + h + h * o + o
    low = 2 if c["bf16"] else 4
    if kind == "predict":
        return {"bytes": 4.0 * r * (i + o) + low * params, "flops": 2.0 * r * (i * h + h * h + h * o)}
    return {"bytes": 4.0 * r * (i + 3 * o) + (4.0 * 7 + low * 2) * params, "flops": 6.0 * r * (i * h + h * h + h * o)}


# ------------------------------------------------------------- FP64 results
def to_real(f):
    """sum_k f(k) e^{i k.x} of half spectra [..., n, n, n/2] (Nyquist modes zero)."""
    n = f.shape[-2]
    return torch.fft.irfftn(torch.nn.functional.pad(f, (0, 1)), s=(n, n, n), dim=(-3, -2, -1), norm="forward")


def to_spec(x):
    n = x.shape[-1]
    f = torch.fft.rfftn(x, dim=(-3, -2, -1), norm="forward")[..., : n // 2].contiguous()
    f[..., n // 2, :, :] = 0
    f[..., :, n // 2, :] = 0
    return f


def exact_orders(d1, n_max, form, cuts):
    """delta_n, theta_n for n = 2..n_max of one realisation (FP64); cuts[n]: |s|
    above it is zero (None: no cut)."""
    n = d1.shape[0]
    s = signed(n).double()
    k = [s[:, None, None], s[None, :, None], torch.arange(n // 2, device="cuda").double()[None, None, :]]
    s2 = s2_grid(n).double()
    inv = torch.where(s2 > 0, 1.0 / s2.clamp(min=1.0), torch.zeros_like(s2))
    d1 = d1.to(torch.complex128)
    orders_k = {1: (d1, d1)}
    fields, out = {}, []
    for m in range(2, n_max + 1):
        dk, tk = orders_k[m - 1]
        phi = tk * inv
        u = [to_real(-1j * k[a] * phi) for a in range(3)]
        if form == "divergence":
            fields[m - 1] = dict(d=to_real(dk), u=u)
        else:
            gd = [to_real(1j * k[a] * dk) for a in range(3)]
            fields[m - 1] = dict(d=to_real(dk), u=u, gd=gd,
                                 t=to_real(tk) if m > 2 else None,
                                 gt=[to_real(1j * k[a] * tk) for a in range(3)] if m > 2 else gd,
                                 du={(a, b): to_real(k[a] * k[b] * phi) for a in range(3) for b in range(a, 3)})
            if m == 2:
                fields[1]["t"] = fields[1]["d"]
        if form == "divergence":
            V = [sum(fields[q]["d"] * fields[m - q]["u"][a] for q in range(1, m)) for a in range(3)]
            S = sum(fields[q]["u"][a] * fields[m - q]["u"][a] for q in range(1, m) for a in range(3))
            A = sum(1j * k[a] * to_spec(V[a]) for a in range(3))
            B = -0.5 * s2 * to_spec(S)
            conv = lambda x: x  # noqa: E731
        else:
            A, B = 0.0, 0.0
            for q in range(1, m):
                f, r = fields[q], fields[m - q]
                A = A + f["d"] * r["t"]
                for a in range(3):
                    A = A + f["gd"][a] * r["u"][a]
                    B = B + f["u"][a] * r["gt"][a]
                for (a, b) in f["du"]:
                    B = B + (1.0 if a == b else 2.0) * f["du"][a, b] * r["du"][a, b]
            conv = to_spec
        c = 2.0 / ((2 * m + 3) * (m - 1))
        new = [conv(c * ((m + 0.5) * A + B)), conv(c * (1.5 * A + m * B))]
        for x in new:
            x[n // 2] = 0
            x[:, n // 2] = 0
            if cuts[m] is not None:
                x[s2 > math.floor(cuts[m] ** 2)] = 0
        orders_k[m] = tuple(new)
        out.append(torch.stack(new))
    return torch.stack(out)


def exact_one(n, n_max, box, batch, seed, form, cuts):
    d = delta1(n, n_max, box, batch, seed)
    return torch.stack([exact_orders(d[b], n_max, form, cuts) for b in range(batch)])


def exact_linear(c, seeds):
    n, box = c["n"], c["box"]
    r = n / (c["n_max"] + 1)
    s2 = s2_grid(n)
    s2[n // 2] = 0
    s2[:, n // 2] = 0
    idx = torch.nonzero((s2 > 0) & (s2 <= math.floor(r * r)))
    s = idx.cpu().numpy().astype(np.int64)
    s[:, :2] = np.where(s[:, :2] < n // 2, s[:, :2], s[:, :2] - n)
    sx, sy, sz = s.T
    sign = np.where((sz > 0) | ((sz == 0) & ((sy > 0) | ((sy == 0) & (sx > 0)))), 1, -1)
    word = ((sx * sign) & 0x1FFFFF) | (((sy * sign) & 0x1FFFFF) << 21) | (((sz * sign) & 0x1FFFFF) << 42)
    amp = np.sqrt(linear_pk(2.0 * math.pi / box * np.sqrt((sx * sx + sy * sy + sz * sz).astype(np.float64))) / box ** 3 / 2.0)
    low = np.uint64(0xFFFFFFFF)
    out = torch.zeros(len(seeds), n, n, n // 2, dtype=torch.complex128, device="cuda")
    for b, seed in enumerate(seeds):
        ctr = [word.astype(np.uint64) & low, word.astype(np.uint64) >> np.uint64(32), np.uint64(0), np.uint64(0)]
        key = [seed & 0xFFFFFFFF, seed >> 32]
        for _ in range(10):   # Philox4x32-10
            p0, p1 = np.uint64(0xD2511F53) * ctr[0], np.uint64(0xCD9E8D57) * ctr[2]
            ctr = [(p1 >> np.uint64(32)) ^ ctr[1] ^ np.uint64(key[0]), p1 & low,
                   (p0 >> np.uint64(32)) ^ ctr[3] ^ np.uint64(key[1]), p0 & low]
            key = [(key[0] + 0x9E3779B9) & 0xFFFFFFFF, (key[1] + 0xBB67AE85) & 0xFFFFFFFF]
        u1, u2 = [(ctr[i].astype(np.float64) + 0.5) * 2.0 ** -32 for i in (0, 1)]
        v = amp * np.sqrt(-2.0 * np.log(u1)) * (np.cos(2 * math.pi * u2) + 1j * sign * np.sin(2 * math.pi * u2))
        out[b, idx[:, 0], idx[:, 1], idx[:, 2]] = torch.from_numpy(v).cuda()
    return out


def exact_power(c, seed):
    d, n, edges = field_set(c, seed, 5), c["n"], torch.tensor(edges_of(c), dtype=torch.float64, device="cuda")
    s2 = s2_grid(n)
    k = 2.0 * math.pi / c["box"] * torch.sqrt(s2.double())
    b = torch.bucketize(k, edges, right=True) - 1
    sel = (b >= 0) & (b < c["nbins"]) & (s2 > 0)
    at = torch.nonzero(sel.reshape(-1))[:, 0]
    bins = b.reshape(-1)[at]
    wt = torch.where(at % (n // 2) == 0, 1.0, 2.0).double()
    cnt = torch.bincount(bins, weights=wt, minlength=c["nbins"])
    out = []
    for i, j in TERMS:
        x, y = (d[q - 1].reshape(-1)[at].to(torch.complex128) for q in (i, j))
        p = torch.bincount(bins, weights=wt * (x * y.conj()).real, minlength=c["nbins"])
        out.append(torch.where(cnt > 0, c["box"] ** 3 * p / cnt.clamp(min=1), torch.zeros_like(p)))
    return torch.stack(out), None


def exact_bispectrum(c, seed):
    d = [f.to(torch.complex128) for f in field_set(c, seed, 4 if c["one_loop"] else 2)]
    n, edges = c["n"], edges_of(c)
    s2 = s2_grid(n)
    k = 2.0 * math.pi / c["box"] * torch.sqrt(s2.double())
    E, N = [], []
    for i in range(c["nbins"]):
        m = ((k >= edges[i]) & (k < edges[i + 1]) & (s2 > 0)).double()
        f = [to_real(x * m) for x in d]
        j3 = (to_real(m.to(torch.complex128)) ** 3).sum()
        if c["one_loop"]:
            t = 6.0 * (f[0] * f[1] * f[2]).sum() + (f[1] ** 3).sum() + 3.0 * (f[0] ** 2 * f[3]).sum()
        else:
            t = (f[0] ** 2 * f[1]).sum()
        nt = j3 / float(n) ** 3
        E.append(torch.where(nt > 0.5, c["box"] ** 6 * t / j3, torch.zeros_like(t)))
        N.append(nt)
    return torch.stack(E), torch.stack(N)


def exact_net(c, seed):
    net = g.MLP(c["n_in"], c["hidden"], c["out"], bf16=c["bf16"], seed=int(seed) % (1 << 31))   # initial weights only
    master = net.master.clone()
    x, t, mask, gen = net_inputs(c, seed)
    i, h, o = c["n_in"], c["hidden"], c["out"]
    low = torch.bfloat16 if c["bf16"] else torch.float32

    def rounded(a):
        return a.float().to(low).double() if c["bf16"] else a

    w = master.to(low).double()
    W1, b1, W2, b2, W3, b3 = (v.reshape(s) for v, s in zip(w.split([i * h, h, h * h, h, h * o, o]),
                                                           [(i, h), (h,), (h, h), (h,), (h, o), (o,)]))
    silu = lambda z: z / (1.0 + torch.exp(-z))  # noqa: E731
    x, t, mask = x.double(), t.double(), mask.double()
    z1 = x @ W1 + b1
    a1 = rounded(silu(z1))
    z2 = a1 @ W2 + b2
    a2 = rounded(silu(z2))
    y = a2 @ W3 + b3
    if c["kind"] == "predict":
        return y
    count = mask.sum()
    loss = (mask * (y - t) ** 2).sum() / count if count > 0 else mask.sum()
    dy = 2.0 * mask * (y - t) / count

    def dsilu(z):
        s = torch.sigmoid(z)
        return s * (1.0 + z * (1.0 - s))

    d2 = (dy @ W3.T) * dsilu(z2)
    d1 = (d2 @ W2.T) * dsilu(z1)
    grad = torch.cat([v.reshape(-1) for v in (x.T @ d1, d1.sum(0), a1.T @ d2, d2.sum(0), a2.T @ dy, dy.sum(0))])
    m, v = net_state(c, gen, master.numel())
    m = 0.9 * m.double() + 0.1 * grad
    v = 0.999 * v.double() + 0.001 * grad * grad
    p = master.double() - 1e-3 * (m / (1.0 - 0.9 ** 101)) / (torch.sqrt(v / (1.0 - 0.999 ** 101)) + 1e-8)
    return dict(y=y, loss=loss.reshape(1), grad=grad, master=p, m=m, v=v, lowp=p)


def exact(c, seed):
    kind = c["kind"]
    if kind == "orders":
        n, n_max = c["n"], c["n_max"]
        if c["truncate"]:      # only the modes below the linear cut are those of the full recursion
            return None
        kc = n / (n_max + 1)
        cuts = [c["cut_nl"] * kc if c["cut_nl"] else None] * (n_max + 1)
        return exact_one(n, n_max, c["box"], c["batch"], seed, c["form"], cuts)
    if kind == "mixed":
        return [exact_one(c["n%d" % i], c["n_max"], c["cell"] * c["n%d" % i], c["batch"], seed * 3 + i, "nine_term",
                          [None] * (c["n_max"] + 1)) for i in range(3)]
    if kind == "linear":
        return exact_linear(c, [int(seed) * 16 + i for i in range(c["batch"])])
    if kind == "power":
        return exact_power(c, seed)
    if kind == "bispectrum":
        return exact_bispectrum(c, seed)
    if kind == "transform":
        gen = generator(seed)
        spec = torch.stack([random_spectrum(c["n"], c["box"], None, gen) for _ in range(c["count"])])
        field = torch.randn(c["count"], c["n"], c["n"], c["n"], generator=gen, device="cuda")
        xs, ks = [], []
        for f in range(c["count"]):
            xs.append(to_real(spec[f].to(torch.complex128)))
            ks.append(to_spec(field[f].double()))
        return torch.stack(xs), torch.stack(ks)
    return exact_net(c, seed)
