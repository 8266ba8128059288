"""What this framework's users have it do: the workloads its speed is judged on.

Three kinds of work, each through the public entry points of
``paper_2111_11687_gb300.nmdose``:

* Monte Carlo dose runs on a phantom whose handle exists (``mc``), on several
  patients in one graph (``patients``) and as whole studies from host buffers
  or from several activity maps (``study``, ``cumulated``);
* the dose denoiser: a training step and whole-volume inference (``train``,
  ``apply``);
* its convolutions, forward and both gradients (``conv``).

Sizes come from the repository's benchmark, tests and experiment: the water
cube, the 8 / 4 / 2 mm adult phantom, uneven patients of 128-256 voxels, the 1
mm whole body, 64^3 patches and the U-Net's channel counts.  Anatomies are the
ones of ``inputs`` (drawn once per grid; above 2^22 voxels at half resolution
and then doubled); CT noise, the PET map and every weight come from the seed.
"""
import functools
import math

import numpy as np
import torch

from paper_2111_11687_gb300 import inputs, nmdose as nm, nuclides

DECAYS = {"18F": nuclides.F18, "18F tracked": nuclides.F18_TRACKED, "177Lu": nuclides.LU177, "131I": nuclides.I131}
FOV = {"adult": (51.2, 51.2, 90.0), "body": (51.2, 51.2, 180.0)}   # cm: grids of other sizes show the same body


# ---- cases -------------------------------------------------------------------
def listed():
    return [
        # the smallest study: the configured count of the point source in water, where launches and the last
        # photons count, not throughput
        dict(name="point_water", kind="mc", body="water", nx=64, ny=64, nz=64, decays=1_000_000, batches=10,
             decay="18F", history=False, read="tally"),
        # the coarse phantom of a quick look (8 mm voxels), maps and organs read back
        dict(name="quick_8mm", kind="mc", body="adult", nx=64, ny=64, nz=75, decays=2_000_000, batches=10,
             decay="18F", history=False, read="maps"),
        # one checkpoint of a run polled until every organ is within 2 %: one batch, organ means only
        dict(name="checkpoint_2mm", kind="mc", body="adult", nx=256, ny=256, nz=300, decays=5_000_000, batches=1,
             decay="18F", history=False, read="organs"),
        # the benchmark step: 1e9 decays on the 2 mm adult phantom, dose and sigma maps
        dict(name="adult_2mm", kind="mc", body="adult", nx=256, ny=256, nz=300, decays=1_000_000_000, batches=10,
             decay="18F", history=False, read="maps"),
        # feet to head at 1 x 1 x 3 mm: the largest grid, at the count that brings its organs to 2 %
        dict(name="whole_body_1mm", kind="mc", body="body", nx=512, ny=512, nz=600, decays=25_000_000, batches=10,
             decay="18F", history=False, read="maps"),
        # the paper's uncertainty method (history by history), positrons tracked, at 4 mm
        dict(name="history_tracked_4mm", kind="mc", body="adult", nx=128, ny=128, nz=150, decays=20_000_000,
             batches=10, decay="18F tracked", history=True, read="maps"),
        # a clinic's list: uneven patients in one graph
        dict(name="patients_8", kind="patients", patients=8, decays=10_000_000, batches=10, side_lo=128, side_hi=256),
        # one patient from the scanner's host buffers to host maps, at the count that satisfies the organ criterion
        dict(name="study_2mm", kind="study", nx=256, ny=256, nz=300, decays=20_000_000),
        # therapy: absorbed dose of 131I from four activity maps, with the radionuclide's own handle
        dict(name="cumulated_131I", kind="cumulated", nx=128, ny=128, nz=150, decays=20_000_000, points=4,
             decay="131I"),
        # one training step of the denoiser at the experiment's size
        dict(name="unet_train", kind="train", patch=64, batch=4, base=16, levels=4),
        # the denoiser on a whole 2 mm map, then the organ means of its result
        dict(name="unet_apply_2mm", kind="apply", nx=256, ny=256, nz=300, roi=False),
        # one convolution layer on its own (a decoder input of level 1), odd-sized: forward, input gradient, weight gradient
        dict(name="conv_96_to_32", kind="conv", n=2, d=50, h=37, w=61, cin=96, cout=32),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["mc", "mc", "mc", "mc", "patients", "study", "cumulated", "train", "apply", "conv"])
    if kind == "mc":
        body = rng.choice(["adult", "adult", "body", "water"])
        if body == "water":
            n = rng.randint(48, 112)
            return dict(kind="mc", body="water", nx=n, ny=n, nz=n, decays=_log(rng, 10**6, 10**8), batches=10,
                        decay="18F", history=False, read="tally")
        side = _log(rng, 60, 400 if body == "body" else 256)
        nz = int(side * rng.uniform(1.0, 1.3))
        decay = rng.choice(["18F", "18F", "18F", "18F tracked", "177Lu", "131I"])
        read = rng.choice(["maps", "maps", "organs", "tally"])
        return dict(kind="mc", body=body, nx=side, ny=side - rng.randint(0, 9), nz=nz,
                    decays=_log(rng, 2 * 10**6, 3 * 10**8), batches=1 if read == "organs" else rng.choice([2, 10, 10, 20]),
                    decay=decay, history=rng.random() < 0.2, read=read)
    if kind == "patients":
        return dict(kind="patients", patients=rng.randint(2, 12), decays=_log(rng, 10**6, 2 * 10**7), batches=10,
                    side_lo=96, side_hi=rng.randint(128, 256))
    if kind == "study":
        side = rng.randint(96, 256)
        return dict(kind="study", nx=side, ny=side - rng.randint(0, 9), nz=rng.randint(120, 300),
                    decays=_log(rng, 5 * 10**6, 2 * 10**8))
    if kind == "cumulated":
        side = rng.randint(64, 200)
        return dict(kind="cumulated", nx=side, ny=side - rng.randint(0, 9), nz=rng.randint(75, 200),
                    decays=_log(rng, 2 * 10**6, 10**8), points=rng.randint(2, 6), decay=rng.choice(["177Lu", "131I"]))
    if kind == "train":
        return dict(kind="train", patch=rng.choice([32, 48, 64]), batch=rng.randint(1, 4), base=16,
                    levels=rng.choice([3, 4, 4]))
    if kind == "apply":
        side = _log(rng, 64, 256)
        return dict(kind="apply", nx=side, ny=side - rng.randint(0, 9), nz=int(side * rng.uniform(1.0, 1.17)),
                    roi=rng.random() < 0.5)
    cout = rng.choice([16, 16, 32, 32, 64, 128])
    edge = 3 if cout < 128 else 8
    return dict(kind="conv", n=rng.randint(1, 4), d=rng.randint(4, 64) // (1 + (cout == 128)) + 2,
                h=rng.randint(8, 192) // edge + 3, w=rng.randint(8, 192) // edge + 3,
                cin=rng.choice([16, 32, 48, 64, 96, 128]) if cout > 16 else rng.choice([16, 48]), cout=cout)


# ---- inputs --------------------------------------------------------------------
def _materials():
    return nm.Materials(inputs.MATERIAL_Z_OVER_A, inputs.MATERIAL_ZEFF, inputs.PE_COEFF, inputs.PE_EXP)


@functools.lru_cache(maxsize=24)
def _anatomy(body, nx, ny, nz):
    """CT numbers, PET means and organ labels [nz, ny, nx] on the GPU, and the voxel size (cm)."""
    f = 2 if nx * ny * nz > 1 << 22 else 1
    shape = tuple(-(-n // f) for n in (nz, ny, nx))
    fov = FOV[body]
    spacing = (fov[0] / nx, fov[1] / ny, fov[2] / nz)
    coarse = tuple(f * s for s in spacing)
    ph = inputs.adult_phantom(shape, coarse, seed=1) if body == "adult" else inputs.whole_body_phantom(shape, coarse, seed=1)
    out = []
    for a in (ph.hu, ph.activity, ph.labels):
        t = torch.from_numpy(a).cuda()
        for axis in range(3) if f > 1 else ():
            t = t.repeat_interleave(f, axis)
        out.append(t[:nz, :ny, :nx].contiguous())
    return out, spacing


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _scan(body, nx, ny, nz, seed):
    """CT (HU, int16), PET (FP32) and labels of one patient: the anatomy with this seed's noise."""
    (hu, act, lab), spacing = _anatomy(body, nx, ny, nz)
    g = _generator(seed)
    noise = torch.randn(hu.shape, generator=g, device="cuda")
    hu = torch.where(act > 0, hu + (10.0 * noise).to(torch.int16), hu)
    act = act * torch.exp(0.2 * torch.randn(hu.shape, generator=g, device="cuda"))
    return hu, act, lab, spacing


def _phantom(hu):
    den = torch.empty(hu.shape, dtype=torch.float32, device="cuda")
    mat = torch.empty(hu.shape, dtype=torch.uint8, device="cuda")
    nm.nm_ct_to_phantom(hu, den, mat)
    return den, mat


def _dose(hu, act, lab, spacing, **kw):
    den, mat = _phantom(hu)
    return nm.Dose(den, mat, spacing, _materials(), activity=act, labels=lab, n_labels=inputs.N_LABELS,
                   activity_bq=inputs.ACTIVITY_BQ, **kw)


def _shape(case):
    return case["nz"], case["ny"], case["nx"]


def _prepare_mc(case, seed):
    s = dict(seed=seed, decays=case["decays"], read=case["read"], history=case["history"])
    shape = _shape(case)
    if case["body"] == "water":
        cube = inputs.water_cube(case["nx"])
        point = np.asarray(cube.point) + np.random.default_rng(seed).uniform(-0.2, 0.2, 3)
        mats = nm.Materials(inputs.WATER_Z_OVER_A, inputs.WATER_ZEFF, inputs.PE_COEFF, inputs.PE_EXP)
        s["d"] = nm.Dose(torch.from_numpy(cube.density).cuda(), torch.from_numpy(cube.material).cuda(), cube.spacing,
                         mats, source_mode=nm.NM_SOURCE_POINT, point=tuple(point), batches=case["batches"])
    else:
        s["d"] = _dose(*_scan(case["body"], case["nx"], case["ny"], case["nz"], seed), batches=case["batches"],
                       history_sigma=int(case["history"]), **DECAYS[case["decay"]])
    if case["read"] == "tally":
        s["tally"] = torch.empty(shape, dtype=torch.int64, device="cuda")
    if case["read"] == "maps":
        s["dose"] = torch.empty(shape, dtype=torch.float32, device="cuda")
        s["sigma"] = torch.empty(shape, dtype=torch.float32, device="cuda")
    if case["history"]:
        s["by_history"] = torch.empty(shape, dtype=torch.float32, device="cuda")
    return s


def _counts(c):
    return np.array([c[k] for k in ("histories", "emitted", "deposited", "escaped", "steps", "compton", "photo", "escapes")],
                    np.int64)


def _run_mc(s):
    d = s["d"]
    d.reset()
    d.run(s["decays"], seed=s["seed"])
    out = {"counts": _counts(d.counters())}
    if s["read"] == "tally":
        nm.nm_dose_get_tally(d.h, s["tally"])
        out["tally"] = s["tally"]
    elif s["read"] == "organs":
        mean, _, _, voxels = d.organs(eps=False, sigma=False)
        out.update(mean=mean, voxels=voxels)
    else:
        d.get(s["dose"], s["sigma"])
        mean, eps, sigma, voxels = d.organs()
        out.update(dose=s["dose"], sigma=s["sigma"], mean=mean, eps=eps, organ_sigma=sigma, voxels=voxels)
    if s["history"]:
        out["by_history"] = d.history_sigma(s["by_history"])
    return out


def _prepare_patients(case, seed):
    r = np.random.default_rng(case["patients"] * 1000 + case["side_hi"])   # the list's grids; the scans are the seed's
    ds = []
    for i in range(case["patients"]):
        side, nz = int(r.integers(case["side_lo"], case["side_hi"] + 1)), int(r.integers(120, 301))
        ds.append(_dose(*_scan("adult", side, side, nz, seed * 100 + i), batches=case["batches"]))
    tallies = [torch.empty(d.shape, dtype=torch.int64, device="cuda") for d in ds]
    return dict(ds=ds, decays=[case["decays"]] * len(ds), seed=seed, tallies=tallies)


def _run_patients(s):
    for d in s["ds"]:
        d.reset()
    nm.nm_dose_run_batch(s["ds"], s["decays"], s["seed"])
    for d, t in zip(s["ds"], s["tallies"]):
        nm.nm_dose_get_tally(d.h, t)
    return {"tally": s["tallies"], "counts": np.stack([_counts(d.counters()) for d in s["ds"]]),
            "mean": np.stack([d.organs(eps=False)[0] for d in s["ds"]])}


def _prepare_study(case, seed):
    hu, act, lab, spacing = _scan("adult", case["nx"], case["ny"], case["nz"], seed)
    pin = lambda t: t.cpu().pin_memory()
    return dict(hu=pin(hu), act=pin(act), lab=pin(lab), spacing=spacing, decays=case["decays"], seed=seed,
                dose=torch.empty(hu.shape).pin_memory(), sigma=torch.empty(hu.shape).pin_memory())


def _run_study(s):
    with _dose(s["hu"], s["act"], s["lab"], s["spacing"]) as d:
        d.run(s["decays"], seed=s["seed"])
        d.get(s["dose"], s["sigma"])
        mean, eps, sigma, voxels = d.organs()
        counts = _counts(d.counters())
    return dict(dose=s["dose"], sigma=s["sigma"], mean=mean, eps=eps, organ_sigma=sigma, voxels=voxels, counts=counts)


def _prepare_cumulated(case, seed):
    hu, act, lab, spacing = _scan("adult", case["nx"], case["ny"], case["nz"], seed)
    den, mat = _phantom(hu)
    g = _generator(seed + 1)
    hours = [2.0 * 2.5**k for k in range(case["points"])]
    half = nuclides.HALF_LIFE_H[case["decay"]]
    maps = [act * 2.0 ** (-t / half) * (0.7 + 0.6 * torch.rand(act.shape, generator=g, device="cuda")) for t in hours]
    return dict(den=den, mat=mat, lab=lab, spacing=spacing, maps=maps, hours=hours, half=half, decays=case["decays"],
                seed=seed, decay=case["decay"], total=torch.empty_like(act), dose=torch.empty_like(act),
                sigma=torch.empty_like(act))


def _run_cumulated(s):
    bq_s = nm.nm_time_integrated_activity(s["maps"], s["hours"], s["half"], s["total"])
    with nm.Dose(s["den"], s["mat"], s["spacing"], _materials(), activity=s["total"], labels=s["lab"],
                 n_labels=inputs.N_LABELS, activity_bq=bq_s, **DECAYS[s["decay"]]) as d:
        d.run(s["decays"], seed=s["seed"])
        d.get(s["dose"], s["sigma"])
        mean, _, sigma, _ = d.organs()
        counts = _counts(d.counters())
    return dict(decays=s["total"], sum=bq_s, dose=s["dose"], sigma=s["sigma"], mean=mean, organ_sigma=sigma,
                counts=counts)


def _exact_cumulated(case, seed):
    s = _prepare_cumulated(case, seed)
    t, a = s["hours"], [m.double() for m in s["maps"]]
    total = a[0] * t[0] / 2
    for k in range(1, len(t)):
        total += (a[k - 1] + a[k]) * (t[k] - t[k - 1]) / 2
    total = 3600.0 * (total + a[-1] * s["half"] / math.log(2.0))
    return dict(decays=total, sum=float(total.sum()), dose=None, sigma=None, mean=None, organ_sigma=None, counts=None)


# The denoiser's parameters as one flat vector: per layer [cout][27 cin padded to a multiple of 128 past 27 cin]
# weights, then the biases, each layer's block padded to 8; the head's weights and bias last.
def _layers(levels, base):
    w, c, out = [base << i for i in range(levels)], 8, []
    for i in range(levels):
        out += [(c, w[i]), (w[i], w[i])]
        c = w[i]
    for i in range(levels - 2, -1, -1):
        out += [(c + w[i], w[i]), (w[i], w[i])]
        c = w[i]
    off, table = 0, []
    for cin, cout in out:
        kpad = (27 * cin + 128) // 128 * 128
        table.append((cin, cout, kpad, off, off + cout * kpad))
        off = (off + cout * kpad + cout + 7) // 8 * 8
    return table, off, (off + base + 1 + 7) // 8 * 8


def _parameters(levels, base, seed):
    """A network in the middle of its training: He-scaled weights, small biases, a head that has left zero."""
    table, head, n = _layers(levels, base)
    r = np.random.default_rng(seed)
    p = np.zeros(n, np.float32)
    for cin, cout, kpad, w, b in table:
        rows = np.zeros((cout, kpad), np.float32)
        rows[:, :27 * cin] = r.normal(0.0, math.sqrt(2.0 / (27 * cin)), (cout, 27 * cin))
        p[w:b] = rows.ravel()
        p[b:b + cout] = r.normal(0.0, 0.02, cout)
    p[head:head + base] = r.normal(0.0, 0.1, base)
    return p


def _network(levels, base, seed):
    d = nm.Denoiser(levels=levels, base_width=base)
    d.params(set=_parameters(levels, base, seed))
    return d


def _prepare_train(case, seed):
    n, p = case["batch"], case["patch"]
    g = _generator(seed)
    smooth = torch.nn.functional.avg_pool3d(torch.rand((n, 4, p, p, p), generator=g, device="cuda"), 5, 1, 2)
    x = torch.zeros((n, p, p, p, 8), dtype=torch.bfloat16, device="cuda")
    x[..., 0] = smooth[:, 0] * (1 + 0.3 * torch.randn((n, p, p, p), generator=g, device="cuda")).clamp(min=0)
    x[..., 1], x[..., 2] = smooth[:, 1] * 2, smooth[:, 2]
    x[..., 3] = smooth[:, 2] / (smooth[:, 1] * 2).clamp(min=0.1)
    net = nm.Denoiser(patch=p, batch=n, levels=case["levels"], base_width=case["base"])
    net.params(set=_parameters(case["levels"], case["base"], seed))
    return dict(net=net, x=x, target=smooth[:, 0].contiguous(), weight=(smooth[:, 3] > 0.45).float(),
                after=torch.empty(net.n_params, device="cuda"), grads=torch.empty(net.n_params, device="cuda"))


def _run_train(s):
    loss = s["net"].train_step(s["x"], s["target"], s["weight"])
    s["net"].params(get=s["after"], grads=s["grads"])
    return dict(loss=loss, weights=s["after"], grads=s["grads"])


def _unet64(x, p, levels, base):
    """The network in 64 bits: x [n, 8, d, h, w], p the flat parameters; y [n, d, h, w]."""
    F = torch.nn.functional
    table, head, _ = _layers(levels, base)

    def conv(t, i):
        cin, cout, kpad, w, b = table[i]
        k = p[w:b].view(cout, kpad)[:, :27 * cin].reshape(cout, 3, 3, 3, cin).permute(0, 4, 1, 2, 3)
        return F.relu(F.conv3d(t, k, p[b:b + cout], padding=1))

    t, skips, i = x, [], 0
    for level in range(levels):
        t = conv(conv(t, i), i + 1)
        i += 2
        if level < levels - 1:
            skips.append(t)
            t = F.avg_pool3d(t, 2)
    while skips:
        t = conv(conv(torch.cat([F.interpolate(t, scale_factor=2, mode="nearest"), skips.pop()], 1), i), i + 1)
        i += 2
    return (t * p[head:head + base].view(1, -1, 1, 1, 1)).sum(1) + p[head + base] + x[:, 0]


def _exact_train(case, seed):
    if case["batch"] * case["patch"]**3 > 1 << 18:
        return None
    s = _prepare_train(case, seed)
    p = torch.from_numpy(_parameters(case["levels"], case["base"], seed)).double().cuda().requires_grad_(True)
    y = _unet64(s["x"].double().permute(0, 4, 1, 2, 3), p, case["levels"], case["base"])
    loss = (s["weight"].double() * (y - s["target"].double()) ** 2).mean()
    loss.backward()
    g = p.grad
    return dict(loss=float(loss.detach()), weights=(p - 1e-3 * g / (g.abs() + 1e-8)).detach(), grads=g)


def _prepare_apply(case, seed):
    hu, act, lab, spacing = _scan("adult", case["nx"], case["ny"], case["nz"], seed)
    d = _dose(hu, act, lab, spacing)
    d.run(10_000_000, seed=seed)
    dose = torch.empty(hu.shape, device="cuda")
    nm.nm_dose_get(d.h, dose)
    den, _ = _phantom(hu)
    return dict(d=d, net=_network(4, 16, seed), dose=dose, den=den, act=act, out=torch.empty_like(dose),
                roi=lab if case["roi"] else None)


def _run_apply(s):
    s["net"].apply(s["dose"], s["den"], s["act"], s["out"], roi=s["roi"])
    return dict(dose=s["out"], mean=s["d"].map_organs(s["out"]))


def _prepare_conv(case, seed):
    n, d, h, w, ci, co = (case[k] for k in ("n", "d", "h", "w", "cin", "cout"))
    g = _generator(seed)
    rand = lambda *s: torch.randn(s, generator=g, device="cuda")
    weights = torch.zeros((co, nm.nm_conv3d_kpad(ci)), dtype=torch.bfloat16, device="cuda")
    weights[:, :27 * ci] = rand(co, 27 * ci) * math.sqrt(2.0 / (27 * ci))
    like = lambda *s: torch.empty(s, dtype=torch.bfloat16, device="cuda")
    return dict(desc=nm._desc(n, d, h, w, ci, cout=co), x=rand(n, d, h, w, ci).relu().bfloat16(),
                dy=(rand(n, d, h, w, co) * 0.1).bfloat16(), w=weights, bias=0.1 * rand(co), y=like(n, d, h, w, co),
                dx=like(n, d, h, w, ci), dw=torch.empty(weights.shape, device="cuda"), db=torch.empty(co, device="cuda"))


def _run_conv(s):
    nm.nm_conv3d_fwd(s["desc"], s["x"], None, s["w"], s["bias"], s["y"], True)
    nm.nm_conv3d_dgrad(s["desc"], s["dy"], s["w"], s["dx"])
    nm.nm_conv3d_wgrad(s["desc"], s["x"], None, s["dy"], s["dw"], s["db"])
    return dict(y=s["y"], dx=s["dx"], dw=s["dw"], db=s["db"])


def _exact_conv(case, seed):
    s = _prepare_conv(case, seed)
    ci, co = case["cin"], case["cout"]
    pad = lambda t: torch.nn.functional.pad(t.double(), (0, 0, 1, 1, 1, 1, 1, 1))
    x, dy, w = pad(s["x"]), pad(s["dy"]), s["w"].double()
    y, dx, dw = s["bias"].double().expand(s["y"].shape).clone(), torch.zeros(s["x"].shape, dtype=torch.float64, device="cuda"), torch.zeros_like(w)
    d, h, wd = case["d"], case["h"], case["w"]
    for tap in range(27):
        z, r, c = tap // 9, tap // 3 % 3, tap % 3
        k = w[:, tap * ci:(tap + 1) * ci]
        xs = x[:, z:z + d, r:r + h, c:c + wd]
        y += xs @ k.T
        dx += dy[:, 2 - z:2 - z + d, 2 - r:2 - r + h, 2 - c:2 - c + wd] @ k
        dw[:, tap * ci:(tap + 1) * ci] = s["dy"].double().reshape(-1, co).T @ xs.reshape(-1, ci)
    return dict(y=y.relu(), dx=dx, dw=dw, db=s["dy"].double().sum((0, 1, 2, 3)))


_PREPARE = dict(mc=_prepare_mc, patients=_prepare_patients, study=_prepare_study, cumulated=_prepare_cumulated,
                train=_prepare_train, apply=_prepare_apply, conv=_prepare_conv)
_RUN = dict(mc=_run_mc, patients=_run_patients, study=_run_study, cumulated=_run_cumulated, train=_run_train,
            apply=_run_apply, conv=_run_conv)
_EXACT = dict(cumulated=_exact_cumulated, train=_exact_train, conv=_exact_conv)


def prepare(case, seed):
    s = _PREPARE[case["kind"]](case, seed)
    s["kind"] = case["kind"]
    return s


def run(state):
    return _RUN[state["kind"]](state)


def exact(case, seed):
    """In 64 bits, what is a plain function of the inputs; a Monte Carlo result is one only of its random numbers."""
    f = _EXACT.get(case["kind"])
    return f(case, seed) if f else None


# Arithmetic a simulated decay cannot do without: per flight step ten Philox rounds (40 operations), a logarithm,
# the move and the voxel test (50); per scatter the angle, the rotation and the new cross sections (120).  An 18F
# decay makes about 14 steps and 3.4 scatters, a photon in water half of that, a 177Lu decay a sixth of a photon.
_PER_DECAY = {"18F": 14 * 90 + 3.4 * 120 + 200, "18F tracked": 14 * 90 + 3.4 * 120 + 400, "131I": 1100, "177Lu": 500}


def work(case):
    k = case["kind"]
    if k in ("mc", "study", "cumulated"):
        v = case["nx"] * case["ny"] * case["nz"]
        if case.get("body") == "water":
            return dict(bytes=5 * v + 8 * v, flops=case["decays"] * (7 * 90 + 1.7 * 120 + 100))
        per = _PER_DECAY[case.get("decay", "18F")]
        maps = {"maps": 8, "tally": 8, "organs": 0}[case.get("read", "maps")]
        grid = {"mc": 9, "study": 7, "cumulated": 10 + 4 * case.get("points", 0)}[k]
        return dict(bytes=v * (grid + maps), flops=case["decays"] * per)
    if k == "patients":
        v = case["patients"] * ((case["side_lo"] + case["side_hi"]) // 2) ** 2 * 210
        return dict(bytes=v * 17, flops=case["patients"] * case["decays"] * _PER_DECAY["18F"])
    if k == "conv":
        m = case["n"] * case["d"] * case["h"] * case["w"]
        return dict(bytes=m * 2 * 2 * (case["cin"] + case["cout"]) + 2 * 27 * case["cin"] * case["cout"] * 4,
                    flops=3 * 2 * m * 27 * case["cin"] * case["cout"])
    levels, base = case.get("levels", 4), case.get("base", 16)
    table, _, n = _layers(levels, base)
    at = [l for l in range(levels) for _ in (0, 1)] + [l for l in range(levels - 2, -1, -1) for _ in (0, 1)]
    per_voxel = sum(2 * 27 * ci * co / 8**l for (ci, co, *_), l in zip(table, at))
    if k == "train":
        m = case["batch"] * case["patch"] ** 3
        return dict(bytes=m * 24 + 20 * n, flops=3 * m * per_voxel)
    v = case["nx"] * case["ny"] * case["nz"]
    body = (0.75 if not case["roi"] else 0.66) * 0.55 * v     # the network's box around the body or the organs
    return dict(bytes=v * 16 + 2 * n, flops=body * per_voxel)
