"""Timed cases of the library: what a user's program calls, over the sizes and
options it is used with.

Every case is one call (or one training step) through the public entry points
on inputs that the program already holds: the sample streams, the output
buffers with their workspace, the descriptors of a batch.  ``exact`` restates
the model in plain 64-bit torch (phase integration, binning, reductions;
gradients by autograd), independent of the library.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2308_09348_gb300 import binding as B
from paper_2308_09348_gb300 import fit as F
from paper_2308_09348_gb300 import inputs as I

MODELS = {"ll": I.MODEL_LL, "qfp": I.MODEL_QFP}
DTYPES = {"f32": torch.float32, "f64": torch.float64}


# ---------------------------------------------------------------------------
# cases
# ---------------------------------------------------------------------------

def _case(kind, n, **kw):
    c = dict(kind=kind, n=int(n), model="qfp", cells=512, precision="f32", weighted=False,
             variant=0, beam="gauss", envelope="gauss", shots=1)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest call: the 32^3 Gauss-Hermite quadrature of a 1 GeV beam
        # with the closed-form classical model, all FP64 (a misalignment scan
        # calls it once per position); latency and launches count
        dict(_case("scatter", 32 ** 3, model="ll", cells=1, precision="f64", weighted=True,
                   beam="hermite"), name="gh32_ll_f64"),
        # Monte Carlo beam, closed-form classical model, every histogram on:
        # reading the samples is what it cannot do without
        dict(_case("scatter", 50_000_003, model="ll", cells=1), name="mc_ll_50m"),
        # the macro-particles of one PIC beam, with their weights, through the
        # quantum model: the interactive prediction
        dict(_case("scatter", 20_011, weighted=True), name="pic_qfp_20k"),
        # the headline workload: 2^26 samples, 512 phase cells
        dict(_case("scatter", 1 << 26), name="mc_qfp_2p26"),
        # the same model in FP64, as used to check an FP32 result
        dict(_case("scatter", 100_003, precision="f64"), name="mc_qfp_f64_100k"),
        # both model refinements on (focus along the path, cycle-averaged
        # quantum factors), an ordinary beam size
        dict(_case("scatter", 524_295, variant=3), name="mc_qfp_refined_500k"),
        # samples that live in pinned host memory (read from a file or made by
        # another program), results back on the host
        dict(_case("host", 4_000_037), name="host_qfp_4m"),
        # a data set of a high-repetition-rate experiment: shots of 1e3 to 1e5
        # samples with their own laser and beam
        dict(_case("batch", 0, shots=400), name="batch_qfp_400"),
        # a delay scan of one beam with the classical model: every shot reads
        # the same samples
        dict(_case("sweep", 100_000, model="ll", cells=1, shots=256), name="sweep_ll_256"),
        # one training step of a parameter fit (forward, loss, adjoint) with
        # the focus taken along the path
        dict(_case("fit", 131_072, variant=1), name="fit_focus_2p17"),
        # one training step of many shots' fits at once, the paper's model
        dict(_case("fit_batch", 1 << 14, shots=64), name="fit_batch_64"),
        # photon spectrum and photon divergence of a beam
        dict(_case("photon", 30_011, bins=256, angles=True), name="photon_30k"),
    ]


def _log_int(rng, lo, hi):
    v = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    return max(lo, min(hi, v | 1 if rng.random() < 0.7 else v))


def draw(rng):
    """One more case of the same ranges."""
    kind = rng.choice(["scatter"] * 5 + ["host", "batch", "batch", "sweep", "fit", "fit",
                                         "fit_batch", "photon"])
    cells = rng.choice([64, 128, 200, 256, 500, 512, 512, 1024])
    weighted = rng.random() < 0.3
    env = rng.choice(["gauss", "gauss", "sin2"])
    if kind == "scatter":
        if rng.random() < 0.4:
            return _case("scatter", _log_int(rng, 5_000, 60_000_000), model="ll", cells=1,
                         precision=rng.choice(["f32", "f32", "f64"]), weighted=weighted,
                         beam=rng.choice(["gauss", "flat"]), envelope=env)
        if rng.random() < 0.25:
            return _case("scatter", _log_int(rng, 5_000, 1 << 17), precision="f64", cells=cells,
                         weighted=weighted, envelope=env)
        return _case("scatter", _log_int(rng, 5_000, 1 << 24), cells=cells, weighted=weighted,
                     beam=rng.choice(["gauss", "flat"]), variant=rng.choice([0, 0, 0, 1, 2, 3]),
                     envelope=env)
    if kind == "host":
        return _case("host", _log_int(rng, 100_000, 8_000_000), cells=cells, weighted=weighted,
                     model=rng.choice(["ll", "qfp"]), envelope=env)
    if kind == "batch":
        return _case("batch", 0, shots=_log_int(rng, 16, 800), cells=cells, weighted=weighted,
                     model=rng.choice(["ll", "qfp", "qfp"]), envelope=env)
    if kind == "sweep":
        return _case("sweep", _log_int(rng, 10_000, 300_000), shots=_log_int(rng, 32, 512),
                     model="ll", cells=1, weighted=weighted, envelope=env)
    if kind == "fit":
        return _case("fit", _log_int(rng, 10_000, 1 << 18), cells=min(cells, 512),
                     weighted=weighted, variant=rng.choice([0, 0, 1, 2]), envelope=env)
    if kind == "fit_batch":
        return _case("fit_batch", _log_int(rng, 2_000, 20_000), shots=_log_int(rng, 8, 64),
                     cells=min(cells, 512), weighted=weighted, envelope=env)
    return _case("photon", _log_int(rng, 2_000, 1 << 16), cells=min(cells, 512),
                 weighted=weighted, bins=rng.choice([100, 128, 256]), angles=rng.random() < 0.5,
                 envelope=env)


# ---------------------------------------------------------------------------
# inputs: descriptors and sample streams, from the case and the seed alone
# ---------------------------------------------------------------------------

def _single(case, seed):
    """Laser, beam and bins of a single-shot case: the library's workload of
    that kind, its laser moved a little (the seed says where)."""
    g = np.random.Generator(np.random.Philox(seed))
    if case["beam"] == "hermite":
        wl = I.tiny_gauss_hermite()
        jx, jy = g.normal(0.0, 1.0, 2)
    else:
        if case["kind"] in ("fit", "fit_batch"):
            wl = I.fit_qfp(1)
        elif case["beam"] == "flat":
            wl = I.broadband_qfp(1)
        else:
            wl = I.full_qfp(1)
        jx, jy = g.normal(0.0, 0.2, 2)
    lz = dict(wl.laser.__dict__)
    lz.update(dx_um=lz["dx_um"] + float(jx), dy_um=lz["dy_um"] + float(jy),
              model=MODELS[case["model"]], variant=case["variant"],
              n_phase=max(case["cells"], 1),
              envelope=I.ENV_GAUSS if case["envelope"] == "gauss" else I.ENV_SIN2)
    return I.Laser(**lz), wl.beam, wl.bins


def _shots(case, seed):
    """Lasers, beams, sample counts and spectrum ranges of a batched case."""
    g = np.random.Generator(np.random.Philox(seed))
    S = case["shots"]
    env = I.ENV_GAUSS if case["envelope"] == "gauss" else I.ENV_SIN2
    common = dict(lambda_um=0.8, tau_fs=30.0, model=MODELS[case["model"]], envelope=env,
                  n_phase=max(case["cells"], 1))
    if case["kind"] == "sweep":
        lz, bm, _ = _single(case, seed)
        delays = np.linspace(-100.0, 100.0, S)
        lasers = [I.Laser(**{**lz.__dict__, "delay_fs": float(d)}) for d in delays]
        hi = 1.2 * bm.gamma_mean * (1 + 4 * bm.rel_spread)
        return lasers, [bm] * S, None, np.array([[0.0, hi]] * S)
    lasers, beams, ranges = [], [], []
    for _ in range(S):
        gm, sp = g.uniform(1e3, 2e4), g.uniform(0.01, 0.2)
        lasers.append(I.Laser(a0=g.uniform(5, 50), w0_um=g.uniform(2, 10), dx_um=g.normal(0, 2),
                              dy_um=g.normal(0, 2), delay_fs=g.normal(0, 30), **common))
        beams.append(I.Beam(gamma_mean=gm, rel_spread=sp, sigma_x_um=3.0, sigma_y_um=3.0,
                            sigma_z_um=10.0, div_rad=1e-3))
        ranges.append((0.0, 1.2 * gm * (1 + 4 * sp)))
    if case["kind"] == "fit_batch":
        counts = np.full(S, case["n"], dtype=np.int64)
    else:
        counts = np.rint(10.0 ** g.uniform(3.0, 5.0, S)).astype(np.int64)
    return lasers, beams, counts, np.array(ranges)


def _streams(case, seed, n, flat):
    """Eight sample streams and the weights, on the GPU."""
    dev = torch.device("cuda")
    dt = DTYPES[case["precision"]]
    g = torch.Generator(device=dev)
    g.manual_seed(seed)
    xi = [torch.randn(n, generator=g, device=dev, dtype=dt) for _ in range(8)]
    if flat:
        xi[3] = torch.rand(n, generator=g, device=dev, dtype=dt)
    w = 0.5 + torch.rand(n, generator=g, device=dev, dtype=dt) if case["weighted"] else None
    return xi, w


def _single_streams(case, seed, flat):
    if case["beam"] == "hermite":
        xi, w = I.gauss_hermite_streams(32)
        dt = DTYPES[case["precision"]]
        return [torch.from_numpy(a).to("cuda", dt) for a in xi], torch.from_numpy(w).to("cuda", dt)
    return _streams(case, seed, case["n"], flat)


def _photon_bins(case):
    return I.Bins(n_bins=case["bins"], lo=1e-3, hi=6720.0, log_spaced=1)


def _batch_bins(case):
    if case["kind"] == "fit_batch":
        return I.Bins(n_bins=256, lo=0.0, hi=1.0, smooth_sigma_bins=2.0)
    return I.Bins(n_bins=512, lo=0.0, hi=1.0)


def _theta(lasers, beams):
    return torch.tensor([[l.a0, l.w0_um, l.dx_um, l.dy_um, l.delay_fs, b.gamma_mean,
                          b.rel_spread, b.div_rad] for l, b in zip(lasers, beams)],
                        dtype=torch.float64)


def _observed(case, theta, ranges, n):
    """The measurement a fit is given, one row per shot: moments and a
    spectrum, a little away from what the starting parameters predict."""
    gm = theta[:, 5]
    nb = 256
    mom = torch.zeros(theta.shape[0], 13, dtype=torch.float64)
    mom[:, 1] = 0.75 * gm                    # mean energy
    mom[:, 2] = 0.12 * gm                    # energy spread
    mom[:, 4] = mom[:, 5] = 1.5e-3           # divergence
    mom[:, 7] = 0.5 * theta[:, 0]            # mean a_eff
    mom[:, 11] = 1.02 * gm                   # mean energy without the laser
    lo, hi = ranges[:, 0], ranges[:, 1]
    centre = lo[:, None] + (torch.arange(nb, dtype=torch.float64) + 0.5) * ((hi - lo) / nb)[:, None]
    S = torch.exp(-0.5 * ((centre - mom[:, 1:2]) / mom[:, 2:3]) ** 2)
    S = S / S.sum(dim=1, keepdim=True) * n
    return mom.cuda(), S.cuda()


def prepare(case, seed):
    """Inputs on the GPU, descriptors, output buffers with their workspace."""
    kind = case["kind"]
    st = dict(case=case)
    if kind in ("batch", "sweep", "fit_batch"):
        lasers, beams, counts, ranges = _shots(case, seed)
        n = case["n"] if counts is None else int(counts.sum())
        st["xi"], st["w"] = _streams(case, seed, n, False)
        off = None if counts is None else np.concatenate([[0], np.cumsum(counts)])
        st["batch"] = B.Batch(lasers, beams, off, _batch_bins(case), n, ranges=ranges,
                              precision=case["precision"])
        if kind == "fit_batch":
            th = _theta(lasers, beams).float()
            st["obs"] = _observed(case, th.double(), torch.from_numpy(ranges), case["n"])
            st["theta"] = th.cuda().requires_grad_(True)
            st["prob"] = F.BatchProblem(st["batch"], st["xi"], st["w"])
        return st
    laser, beam, bins = _single(case, seed)
    st.update(laser=laser, beam=beam, bins=bins)
    st["xi"], st["w"] = _single_streams(case, seed, bool(beam.flat_energy))
    if kind == "scatter":
        st["out"] = B.Outputs(bins, case["n"], precision=case["precision"])
    elif kind == "host":
        st["xi"] = [x.cpu().pin_memory() for x in st["xi"]]
        st["w"] = None if st["w"] is None else st["w"].cpu().pin_memory()
        st["out"] = B.HostOutputs(bins, st["xi"], st["w"], precision=case["precision"])
    elif kind == "photon":
        pb = st["bins"] = _photon_bins(case)
        st["out"] = torch.zeros(pb.n_bins, dtype=torch.float64, device="cuda")
        st["theta2"] = (torch.zeros(2, pb.n_bins, dtype=torch.float64, device="cuda")
                        if case["angles"] else None)
        st["work"] = torch.empty(64 << 20, dtype=torch.uint8, device="cuda")
    elif kind == "fit":
        th = _theta([laser], [beam]).float()
        obs = _observed(case, th.double(), torch.tensor([[bins.lo, bins.hi]], dtype=torch.float64),
                        case["n"])
        st["obs"] = tuple(t[0] for t in obs)
        st["prob"] = F.Problem(laser, beam, bins, st["xi"], st["w"],
                               out=B.Outputs(bins, case["n"]))
        # the parameters in torch's default type, as a training script has them
        st["theta"] = th[0].clone().requires_grad_(True)
    return st


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "scatter":
        o = B.qs_scatter(st["laser"], st["beam"], st["xi"], st["bins"], w=st["w"],
                         precision=case["precision"], out=st["out"])
        return _single_outputs(o)
    if kind == "host":
        o = B.qs_scatter_host(st["laser"], st["beam"], st["xi"], st["bins"], w=st["w"],
                              precision=case["precision"], out=st["out"])
        return _single_outputs(o)
    if kind in ("batch", "sweep"):
        b = st["batch"].run(st["xi"], st["w"])
        return {"spectra": b.spectra, "moments": b.moments}
    if kind == "photon":
        r = B.qs_photon_spectrum(st["laser"], st["beam"], st["xi"], st["bins"], w=st["w"],
                                 out=st["out"], theta2=st["theta2"], workspace=st["work"])
        return {"spectrum": r[0], "theta2": r[1]} if case["angles"] else {"spectrum": r}
    theta = st["theta"]
    theta.grad = None
    if kind == "fit":
        mom, S = F.ScatterFn.apply(theta, st["prob"])
        loss = F.loss_fn(mom, S, *st["obs"], F.DEFAULT_MOMENT_WEIGHTS, 1.0)
    else:
        mom, S = F.BatchScatterFn.apply(theta, st["prob"])
        loss = F.loss_batch(mom, S, *st["obs"], F.BATCH_MOMENT_WEIGHTS, 1.0).sum()
    loss.backward()
    return {"moments": mom.detach(), "smooth": S.detach(), "grad": theta.grad}


def _single_outputs(o):
    return {"spectrum": o.spectrum, "divmap": o.divmap, "aeff": o.aeff_hist,
            "moments": o.moments}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

# Operations (an add, a product, a quotient, a logarithm, an exponential each
# counting one) of the model as it is written: decode, focus and closed form
# of one sample; one phase cell of the quantum model, and what the focus along
# the path adds to it; one photon-energy bin of one cell of one sample.
OPS_SAMPLE, OPS_CELL, OPS_CELL_FOCUS, OPS_PHOTON = 60, 75, 22, 30


def work(case):
    kind, esz = case["kind"], 4 if case["precision"] == "f32" else 8
    qfp = case["model"] == "qfp"
    cell = OPS_CELL + (OPS_CELL_FOCUS if case["variant"] & I.VAR_CELL_FOCUS else 0)
    streams = (8 if qfp else 6) + (1 if case["weighted"] else 0)
    shots = case["shots"]
    if kind == "batch":
        n = evals = int(shots * (1e5 - 1e3) / math.log(100.0))
    elif kind == "sweep":
        n, evals = case["n"], case["n"] * shots
    else:
        n = evals = case["n"] * shots
    if kind == "photon":
        streams = 6 + (1 if case["weighted"] else 0)
        flops = evals * (OPS_SAMPLE + case["cells"] * (cell + case["bins"] * OPS_PHOTON))
        return {"bytes": n * streams * esz + 24 * case["bins"], "flops": flops}
    flops = evals * (OPS_SAMPLE + (case["cells"] * cell if qfp else 0))
    out = 8 * 13 * shots
    if kind in ("scatter", "host"):
        b = _single(case, 0)[2]
        out += 8 * (b.n_bins + b.n_tx * b.n_ty + b.n_aeff)
    else:
        out += 8 * 512 * shots
    if kind in ("fit", "fit_batch"):
        # the adjoint reads the samples again and carries two tangents
        return {"bytes": 2 * n * streams * esz + out, "flops": 3 * flops}
    return {"bytes": n * streams * esz + out, "flops": flops}


# ---------------------------------------------------------------------------
# the model in 64 bits
# ---------------------------------------------------------------------------

LN2 = math.log(2.0)
C_LIGHT = 0.299792458
R_E, LBAR_C = 2.8179403262e-9, 3.8615926796e-7
ALPHA = 7.2973525693e-3
KAPPA = math.sqrt(2.0 / math.pi)
EXACT_EVALS = 3e10        # sample-cells that take some seconds in 64 bits


def _gaunt(x):
    L = torch.log1p(1.7 * x)
    r = 1.0 / (1.0 + 1.7 * x)
    Bq = 1.0 + 4.8 * (1.0 + x) * L + 2.44 * x * x
    B1 = 4.8 * L + 8.16 * (1.0 + x) * r + 4.88 * x
    g = Bq ** (-2.0 / 3.0)
    chig1 = (-2.0 / 3.0) * g / Bq * B1 * x
    h = g * (1.0 + 4.26 * x + 0.494 * x * x) / (1.0 + x * (12.32 + x * (17.44 + 1.63 * x)))
    return g, 2.0 * g + chig1, h


NODES = 1 << 16


def _lookup(tab, x):
    """Four-point Lagrange interpolation of the rows of tab at coordinate x."""
    i = x.detach().floor().clamp(1, tab[0].numel() - 3).long()
    t = x - i
    c = [-t * (t - 1) * (t - 2) / 6, (t + 1) * (t - 1) * (t - 2) / 2,
         -(t + 1) * t * (t - 2) / 2, (t + 1) * t * (t - 1) / 6]
    return [sum(c[k] * v[i + (k - 1)] for k in range(4)) for v in tab]


CYC_U, CYC_S = 16.0, 0.02


@functools.lru_cache(maxsize=1)
def _cycle_table():
    """Means over the laser cycle of the three rate factors on a dense grid of
    log2(1 + chi/0.02)."""
    z, w = np.polynomial.legendre.leggauss(128)
    c = torch.from_numpy(np.cos(0.25 * math.pi * (1 + z))).cuda()
    w = torch.from_numpy(0.5 * w).cuda()
    u = torch.arange(NODES, dtype=torch.float64, device="cuda") * (CYC_U / (NODES - 1))
    chi = CYC_S * (torch.exp2(u) - 1.0)
    g, s, h = _gaunt(math.sqrt(2.0) * chi[:, None] * c)
    wc = w * 2.0 * c * c
    # chi dG/dchi = <2 cos^2 x g'(x)>, so S = <2 cos^2 (2g + x g')>
    return [(wc * g).sum(1), (wc * s).sum(1), (wc * math.sqrt(2.0) * c * h).sum(1)]


def _factors(chi, variant):
    if variant & I.VAR_CYCLE_CHI:
        u = torch.log2(1.0 + chi / CYC_S)
        return _lookup(_cycle_table(), u * ((NODES - 1) / CYC_U))
    return _gaunt(chi)


PH_LO, PH_HI = -60.0, 6.2


@functools.lru_cache(maxsize=1)
def _bessel_table():
    """K_{2/3}(y) e^y y^(2/3) and int_y K_{1/3} e^y on a dense grid of log2 y."""
    out = [[], []]
    t = torch.arange(2400, dtype=torch.float64, device="cuda") / 40.0
    wt = torch.full_like(t, 1.0 / 40.0)
    wt[0] *= 0.5
    ch = torch.cosh(t)
    for u in torch.linspace(PH_LO, PH_HI, NODES, dtype=torch.float64, device="cuda").split(8192):
        y = torch.exp2(u)[:, None]
        e = torch.exp(-y * (ch - 1.0)) * wt
        out[0].append((e * torch.cosh(2.0 * t / 3.0)).sum(1) * y[:, 0] ** (2.0 / 3.0))
        out[1].append((e * torch.cosh(t / 3.0) / ch).sum(1))
    return [torch.cat(o) for o in out]


class _Model:
    """One case's laser window and its samples' records in 64 bits."""

    def __init__(self, case, laser, beam):
        self.case, self.bm = case, beam
        self.k = 2.0 * math.pi / laser.lambda_um
        self.lam = laser.lambda_um
        self.Rc = R_E * self.k
        self.cchi = math.sqrt(2.0) * self.k * LBAR_C
        Phi = C_LIGHT * self.k * laser.tau_fs
        N = max(case["cells"], 1)
        j = np.arange(N) + 0.5
        if case["envelope"] == "gauss":
            self.h = 5.0 * Phi / N
            phi = -2.5 * Phi + j * self.h
            self.G = np.exp(-2.0 * LN2 * (phi / Phi) ** 2)
            self.shift = phi / (2.0 * self.k)
            self.intG2 = Phi * math.sqrt(math.pi / (4.0 * LN2))
        else:
            PhiT = Phi / (1.0 - 2.0 / math.pi * math.asin(2.0 ** -0.25))
            self.h = PhiT / N
            phi = j * self.h
            self.G = np.sin(math.pi * phi / PhiT) ** 2
            self.shift = (phi - 0.5 * PhiT) / (2.0 * self.k)
            self.intG2 = 3.0 * PhiT / 8.0

    def front(self, th, xi):
        """Decode and crossing geometry; th: 8 parameters (per sample or one)."""
        b = self.bm
        a0, w0, dx, dy, delay, gm, sp, div = th
        x, y = b.dx_um + b.sigma_x_um * xi[0], b.dy_um + b.sigma_y_um * xi[1]
        z = b.sigma_z_um * xi[2]
        if b.flat_energy:
            g0 = b.gamma_lo + (b.gamma_hi - b.gamma_lo) * xi[3]
        else:
            g0 = gm * (1.0 + sp * xi[3])
        g0 = torch.clamp(g0, min=1.0)
        thx, thy = div * xi[4], div * xi[5]
        cd = C_LIGHT * delay
        ct, zs = 0.5 * (z + cd), 0.5 * (z - cd)
        xs, ys = x + thx * ct - dx, y + thy * ct - dy
        return dict(a0=a0, w0=w0, zR=math.pi * w0 * w0 / self.lam, g0=g0, thx=thx, thy=thy,
                    zs=zs, xs=xs, ys=ys)

    def amp(self, f, s=0.0):
        q = 1.0 + ((f["zs"] - s) / f["zR"]) ** 2
        rho2 = (f["xs"] + f["thx"] * s) ** 2 + (f["ys"] + f["thy"] * s) ** 2
        return f["a0"] * q ** -0.5 * torch.exp(-rho2 / (f["w0"] ** 2 * q))

    def cells(self, f):
        """Every phase cell's (field amplitude, mu, chi); the last state is
        left in f (du, V)."""
        focus = self.case["variant"] & I.VAR_CELL_FOCUS
        g0, a = f["g0"], self.amp(f)
        du = torch.zeros_like(g0)
        V = torch.zeros_like(g0)
        gprev = 1.0
        K0 = 2.0 / 3.0 * self.Rc
        c55 = 55.0 / (16.0 * math.sqrt(3.0))
        for G, s in zip(self.G.tolist(), self.shift.tolist()):
            A = (self.amp(f, s) if focus else a) * G
            hK = self.h * K0 * A * A
            mu = g0 / (1.0 + g0 * (du + 0.5 * hK * gprev))
            chi = self.cchi * mu * A
            yield A, mu, chi
            g, sf, h2 = _factors(chi, self.case["variant"])
            du = du + hK * g
            lam = -2.0 * hK * mu * sf
            r = lam * V + c55 * hK * mu ** 3 * chi * h2
            V = V + r * (1.0 + 0.5 * lam)
            gprev = g
        f["du"], f["V"] = du, V

    def records(self, th, xi):
        f = self.front(th, xi)
        a, g0 = self.amp(f), f["g0"]
        if self.case["model"] == "ll":
            mu = g0 / (1.0 + 2.0 / 3.0 * self.Rc * self.intG2 * g0 * a * a)
            z = torch.zeros_like(mu)
            return dict(g0=g0, a=a, mu=mu, V=z, te=z, gout=mu, tx=f["thx"], thx=f["thx"],
                        thy=f["thy"])
        for _ in self.cells(f):
            pass
        mu, V = g0 / (1.0 + g0 * f["du"]), f["V"]
        sv = torch.sqrt(V.clamp_min(1e-300))
        te = KAPPA * a * sv / (mu * mu)
        return dict(g0=g0, a=a, mu=mu, V=V, te=te, gout=mu + sv * xi[7],
                    tx=f["thx"] + te * xi[6], thx=f["thx"], thy=f["thy"])


def _sums(r, w, shot, S):
    """The sums that the moments come from, one row per shot."""
    rows = [w, w * r["mu"], w * r["V"], w * (r["thx"] ** 2 + r["te"] ** 2), w * r["thy"] ** 2,
            w * r["a"], w * r["g0"]]
    z = torch.zeros(S, dtype=torch.float64, device=w.device)
    return torch.stack([z.index_add(0, shot, x) for x in rows], dim=1)


def _moments(s, M2):
    W = s[:, 0]
    mean = s[:, 1] / W
    spread = torch.sqrt((M2 + s[:, 2]) / W)
    dx, dy = torch.sqrt(s[:, 3] / W), torch.sqrt(s[:, 4] / W)
    z = torch.zeros_like(W)
    return torch.stack([W, mean, spread, spread / mean, dx, dy,
                        torch.sqrt((s[:, 3] + s[:, 4]) / W), s[:, 5] / W, z, z, z, s[:, 6] / W, z],
                       dim=1)


def _hist(idx, w, size):
    return torch.bincount(idx, weights=w, minlength=size)[:size]


def _pieces(n, step):
    return [slice(i, min(n, i + step)) for i in range(0, n, step)]


def _exact_shots(case, model, theta, ranges, bins, streams, w, counts):
    """Spectra (with under and over), moments; maps where the bins have them."""
    S, dev = theta.shape[0], "cuda"
    n = streams[0].numel()
    if counts is None and S > 1:                # every shot reads every sample
        parts = [_exact_shots(case, model, theta[s:s + 1], ranges[s:s + 1], bins, streams, w, None)
                 for s in range(S)]
        return {k: torch.cat([p[k] for p in parts]) for k in ("spectra", "moments")}
    off = torch.tensor([0, n] if counts is None else [0, *np.cumsum(counts)], device=dev)
    nb = bins.n_bins
    spec = torch.zeros(S * (nb + 2), dtype=torch.float64, device=dev)
    nmap = bins.n_tx * bins.n_ty
    dmap = torch.zeros(nmap + 1, dtype=torch.float64, device=dev)
    ahist = torch.zeros(bins.n_aeff + 1, dtype=torch.float64, device=dev)
    sums = torch.zeros(S, 7, dtype=torch.float64, device=dev)
    ref = theta[:, 5].cuda() if not model.bm.flat_energy else torch.full((S,), 1e4, device=dev)
    M2 = torch.zeros(S, 2, dtype=torch.float64, device=dev)
    lo, hi = ranges[:, 0].cuda(), ranges[:, 1].cuda()
    for p in _pieces(n, 1 << 22):
        xi = [x[p].double() for x in streams]
        m = xi[0].numel()
        ww = torch.ones(m, dtype=torch.float64, device=dev) if w is None else w[p].double()
        if S == 1:
            shot = torch.zeros(m, dtype=torch.long, device=dev)
            th = theta[0].tolist()
        else:
            shot = torch.searchsorted(off, torch.arange(p.start, p.stop, device=dev),
                                      right=True) - 1
            th = [theta[:, k].cuda()[shot] for k in range(8)]
        r = model.records(th, xi)
        sums += _sums(r, ww, shot, S)
        d = r["mu"] - ref[shot]
        M2[:, 0].index_add_(0, shot, ww * d)
        M2[:, 1].index_add_(0, shot, ww * d * d)
        if bins.log_spaced:
            t = torch.log(r["gout"].clamp_min(1e-300) / lo[shot]) * nb / torch.log(hi / lo)[shot]
        else:
            t = (r["gout"] - lo[shot]) * nb / (hi - lo)[shot]
        k = torch.where(t < 0, nb, torch.where(t >= nb, nb + 1, t.floor())).long()
        spec += _hist(shot * (nb + 2) + k, ww, S * (nb + 2))
        if nmap:
            fx = ((r["tx"] + bins.theta_max) * bins.n_tx / (2 * bins.theta_max)).floor()
            fy = ((r["thy"] + bins.theta_max) * bins.n_ty / (2 * bins.theta_max)).floor()
            ok = (fx >= 0) & (fx < bins.n_tx) & (fy >= 0) & (fy < bins.n_ty)
            dmap += _hist(torch.where(ok, fy * bins.n_tx + fx, nmap).long(), ww, nmap + 1)
        if bins.n_aeff:
            ka = (r["a"] * bins.n_aeff / bins.aeff_max).floor().clamp(max=bins.n_aeff).long()
            ahist += _hist(ka, ww, bins.n_aeff + 1)
    spec = spec.view(S, nb + 2)
    mom = _moments(sums, M2[:, 1] - M2[:, 0] ** 2 / sums[:, 0])
    mom[:, 8], mom[:, 9] = spec[:, nb], spec[:, nb + 1]
    mom[:, 10] = dmap[nmap]
    return {"spectra": spec[:, :nb].contiguous(), "moments": mom, "divmap": dmap[:nmap],
            "aeff": ahist[:bins.n_aeff]}


def _exact_fit(case, model, theta, ranges, bins, streams, w, counts, obs):
    """Moments, smoothed spectra and the loss's gradient, by autograd over
    pieces of the samples (the loss sees sums over all of them: one pass for
    the sums, one for the gradient)."""
    S, dev = theta.shape[0], "cuda"
    n, nb, sg = streams[0].numel(), bins.n_bins, bins.smooth_sigma_bins
    th0 = theta.cuda().clone().requires_grad_(True)
    lo, hi = ranges[:, 0].cuda(), ranges[:, 1].cuda()
    off = torch.tensor([0, *np.cumsum(counts)], device=dev)

    def part(p, ref):
        xi = [x[p].double() for x in streams]
        ww = (torch.ones(xi[0].numel(), dtype=torch.float64, device=dev) if w is None
              else w[p].double())
        shot = torch.searchsorted(off, torch.arange(p.start, p.stop, device=dev), right=True) - 1
        r = model.records([th0[:, k][shot] for k in range(8)], xi)
        s = _sums(r, ww, shot, S)
        q = torch.zeros(S, dtype=torch.float64, device=dev)
        d = r["mu"] - ref[shot]
        q = torch.stack([q.index_add(0, shot, ww * d), q.index_add(0, shot, ww * d * d)], dim=1)
        t = (r["gout"] - lo[shot]) * nb / (hi - lo)[shot]
        half = int(math.ceil(6 * sg)) + 1
        k = t.detach().floor().long()[:, None] + torch.arange(-half, half + 1, device=dev)
        e = k + 0.5 - t[:, None]
        on = (e.detach().abs() <= 6 * sg) & (k >= 0) & (k < nb)
        v = torch.where(on, ww[:, None] * torch.exp(-e * e / (2 * sg * sg)), 0.0)
        v = v / (sg * math.sqrt(2 * math.pi))
        sm = torch.zeros(S * nb, dtype=torch.float64, device=dev)
        sm = sm.index_add(0, (shot[:, None] * nb + k.clamp(0, nb - 1)).reshape(-1), v.reshape(-1))
        return s, q, sm.view(S, nb), r["gout"].detach(), ww, shot

    ref = th0.detach()[:, 5]
    steps = _pieces(n, 1 << 17)
    tot, counted = None, torch.zeros(S, 2, dtype=torch.float64, device=dev)
    with torch.no_grad():
        for p in steps:
            *v, gout, ww, shot = part(p, ref)
            tot = v if tot is None else [x + y for x, y in zip(tot, v)]
            counted[:, 0].index_add_(0, shot, torch.where(gout < lo[shot], ww, 0.0))
            counted[:, 1].index_add_(0, shot, torch.where(gout >= hi[shot], ww, 0.0))
    tot = [t.clone().requires_grad_(True) for t in tot]
    mom = _moments(tot[0], tot[1][:, 1] - tot[1][:, 0] ** 2 / tot[0][:, 0])
    mw = F.DEFAULT_MOMENT_WEIGHTS if case["kind"] == "fit" else F.BATCH_MOMENT_WEIGHTS
    tm, tS = (t.reshape(S, -1) for t in obs)
    loss = (((tot[2] - tS) / tS.sum(1, keepdim=True)) ** 2).sum() * nb
    for name, c in mw.items():
        i = F.MOMENT_INDEX[name]
        loss = loss + (c * ((mom[:, i] - tm[:, i]) / tm[:, i].abs()) ** 2).sum()
    up = torch.autograd.grad(loss, tot)
    for p in steps:
        v = part(p, ref)[:3]
        torch.autograd.backward(v, up)
    mom = mom.detach()
    mom[:, 8:10] = counted
    return {"moments": mom, "smooth": tot[2].detach(), "grad": th0.grad}


def _exact_photon(case, model, theta, bins, streams, w):
    nb = bins.n_bins
    eps = bins.lo * (bins.hi / bins.lo) ** ((torch.arange(nb, dtype=torch.float64, device="cuda")
                                             + 0.5) / nb)
    tab = _bessel_table()
    pref = model.h * ALPHA / (2 * math.sqrt(3.0) * math.pi) * math.sqrt(2.0) / model.cchi
    out = torch.zeros(3, nb, dtype=torch.float64, device="cuda")
    for p in _pieces(streams[0].numel(), 1 << 15):
        xi = [x[p].double() for x in streams]
        f = model.front(theta[0].tolist(), xi)
        ww = torch.ones_like(f["g0"]) if w is None else w[p].double()
        for A, mu, chi in model.cells(f):
            xr = eps / mu[:, None]
            om = 1.0 - xr
            y = 2.0 * xr / (3.0 * chi[:, None] * om)
            on = (om > 0) & (y < 60.0)
            y = torch.where(on, y, 1.0)
            om = torch.where(on, om, 1.0)
            k23, ki13 = _lookup(tab, (torch.log2(y).clamp_min(PH_LO) - PH_LO)
                                * ((NODES - 1) / (PH_HI - PH_LO)))
            Fq = torch.exp(-y) * ((om + 1.0 / om) * k23 * y ** (-2.0 / 3.0) - ki13)
            c = pref * ww / (mu * mu)
            ax = f["thx"] ** 2 + (0.5 * A * A + 1.0) / (mu * mu)
            ay = f["thy"] ** 2 + 1.0 / (mu * mu)
            out += torch.stack([c, c * ax, c * ay]) @ torch.where(on, Fq, 0.0)
    return {"spectrum": out[0], "theta2": out[1:]} if case["angles"] else {"spectrum": out[0]}


def exact(case, seed):
    kind = case["kind"]
    cells = case["cells"] if case["model"] == "qfp" else 1
    if kind != "batch" and case["n"] * case["shots"] * cells > EXACT_EVALS:
        return None
    with torch.no_grad():
        if kind in ("batch", "sweep", "fit_batch"):
            lasers, beams, counts, ranges = _shots(case, seed)
            n = case["n"] if counts is None else int(counts.sum())
            streams, w = _streams(case, seed, n, False)
            laser, beam, bins = lasers[0], beams[0], _batch_bins(case)
            theta, ranges = _theta(lasers, beams), torch.from_numpy(ranges)
        else:
            laser, beam, bins = _single(case, seed)
            streams, w = _single_streams(case, seed, bool(beam.flat_energy))
            counts, theta = [case["n"]], _theta([laser], [beam])
            ranges = torch.tensor([[bins.lo, bins.hi]], dtype=torch.float64)
        model = _Model(case, laser, beam)
        if kind == "photon":
            return _exact_photon(case, model, theta, _photon_bins(case), streams, w)
        if kind not in ("fit", "fit_batch"):
            r = _exact_shots(case, model, theta, ranges, bins, streams, w, counts)
            if kind in ("batch", "sweep"):
                return {"spectra": r["spectra"], "moments": r["moments"]}
            return {"spectrum": r["spectra"][0], "divmap": r["divmap"], "aeff": r["aeff"],
                    "moments": r["moments"][0]}
        theta = theta.float().double()
        obs = _observed(case, theta, ranges, case["n"])
    r = _exact_fit(case, model, theta, ranges, bins, streams, w, counts, obs)
    return {k: v[0] for k, v in r.items()} if kind == "fit" else r
