"""Performance cases: the calls a Reinforced Dynamics run makes of this library.

One RiD iteration explores with a biased ensemble, selects frames, labels them
with restrained (or constrained) runs, trains the ensemble on the labels and
projects it by MCMC.  The listed cases are those calls at the sizes of the
repository's workloads and benchmark; `draw` gives the same calls over the
ranges of chain lengths, walker counts, network shapes and precisions that the
configurations, the batching and serving mixes and the tests use.

Runs that follow a trajectory are short (10 to 200 steps): molecular dynamics is
chaotic, and a longer call repeats the same step.
"""
import math

import numpy as np
import torch

from paper_2408_14070_gb300 import inputs as I
from paper_2408_14070_gb300 import rid

PRECISION = {"fp32": rid.RID_PREC_FP32, "bf16": rid.RID_PREC_BF16, "fp8": rid.RID_PREC_FP8}
F64 = torch.float64
# what exact() may spend: multiply-adds of the 64-bit networks, and chain pairs
EXACT_FLOPS, EXACT_PAIRS = 6e12, 4e9


def listed():
    return [
        # the smallest exploration: a 22-bead chain, 16 walkers, a small FP32 ensemble
        dict(name="explore_tiny", kind="explore", beads=22, cvs=2, walkers=16, models=4, layers=3, width=64,
             resnet=False, precision="fp32", steps=200),
        # the paper's own network (residual, width 300) at its 12 walkers: latency per step
        dict(name="explore_paper_w12", kind="explore", beads=200, cvs=18, walkers=12, models=4, layers=4, width=300,
             resnet=True, precision="bf16", steps=100),
        # the benchmark's workload: 1024 walkers on the 200-bead chain, BF16 ensemble
        dict(name="explore_n200_w1024", kind="explore", beads=200, cvs=20, walkers=1024, models=4, layers=4, width=256,
             resnet=False, precision="bf16", steps=50),
        # the largest: 8192 walkers, eight wide members
        dict(name="explore_n100_w8192", kind="explore", beads=100, cvs=32, walkers=8192, models=8, layers=4, width=512,
             resnet=False, precision="bf16", steps=10),
        # one force evaluation with every output, plain FP32 ensemble
        dict(name="forces_fp32_w1024", kind="forces", beads=200, cvs=20, walkers=1024, models=4, layers=4, width=256,
             resnet=False, precision="fp32"),
        # restrained labels of one iteration's selected frames (30 in the paper's selector settings)
        dict(name="label_r30", kind="label", beads=200, cvs=20, runs=30, steps=100),
        # 512 uneven restrained labeling jobs in one call, from host arrays
        dict(name="label_batch_512", kind="label_batch", jobs=512, beads_lo=50, beads_hi=500, cvs_lo=4, cvs_hi=40,
             mix=3, steps=250),
        # constrained labels on distance CVs
        dict(name="constrained_r1024", kind="constrained", beads=200, pairs=10, runs=1024, steps=50),
        # Adam steps of the exploration model on 16384 labels, batch 128 and dropout 0.1 as in the paper
        dict(name="train_4x256", kind="train", cvs=20, models=4, layers=4, width=256, resnet=False, batch=128,
             dropout=0.1, labels=16384, steps=20),
        # dimension reduction of the trained ensemble, FP32, the paper's 2000 walkers and 101 bins
        dict(name="mcmc_fp32_w2000", kind="mcmc", cvs=20, models=4, layers=4, width=256, resnet=False, walkers=2000,
             steps=50, bins=101),
        # the same walk through a system's BF16 ensemble
        dict(name="mcmc_bf16_w2000", kind="mcmc_system", cvs=20, models=4, layers=4, width=256, resnet=False,
             precision="bf16", walkers=2000, steps=100, bins=101),
        # selection on the traces of 1024 walkers x 100 frames, threshold adapted into 30-45 clusters
        dict(name="select_102k", kind="select", frames=102400, cvs=20, threshold=2.6, lower=30, upper=45,
             max_selection=50),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _capped_steps(rng, lo, hi, per_step, most):
    """Log-uniform in [lo, hi], lowered so that the run costs at most `most`."""
    return max(lo, min(_log(rng, lo, hi), int(most / max(per_step, 1.0))))


def draw(rng):
    kind = rng.choice(["explore", "explore", "explore", "explore", "forces", "label", "label_batch", "constrained",
                       "train", "mcmc", "mcmc_system", "select"])
    net = dict(models=rng.choice([2, 4, 4, 8]), layers=rng.choice([2, 3, 4, 4]), width=_log(rng, 48, 512),
               resnet=rng.random() < 0.4)
    if kind in ("explore", "forces"):
        beads = _log(rng, 20, 600)
        cvs = rng.randint(2, min(40, beads - 3))
        walkers = _log(rng, 4, 4096)
        c = dict(kind=kind, beads=beads, cvs=cvs, walkers=walkers, **net,
                 precision=rng.choice(["fp32", "bf16", "bf16", "fp8"]))
        per = _mlp_flops(c) * (20.0 if c["precision"] == "fp32" else 1.0) * walkers
        pair = 20.0 * walkers * beads * beads
        c["walkers"] = max(4, int(walkers * min(1.0, 4e11 / per, 4e10 / pair)))
        if kind == "explore":
            scale = c["walkers"] / walkers
            c["steps"] = _capped_steps(rng, 5, 200, (per + 10.0 * pair) * scale, 1.2e12)
        return c
    if kind == "label":
        beads = _log(rng, 20, 1000)
        runs = max(1, min(_log(rng, 1, 300), int(1.2e7 / beads ** 2)))
        return dict(kind=kind, beads=beads, cvs=rng.randint(2, min(40, beads - 3)), runs=runs,
                    steps=rng.randint(40, 120))
    if kind == "label_batch":
        lo = _log(rng, 24, 100)
        return dict(kind=kind, jobs=_log(rng, 16, 512), beads_lo=lo, beads_hi=rng.randint(lo + 20, 500), cvs_lo=2,
                    cvs_hi=rng.randint(4, 40), mix=rng.randint(1, 10 ** 6), steps=rng.randint(40, 250))
    if kind == "constrained":
        beads = _log(rng, 40, 400)
        return dict(kind=kind, beads=beads, pairs=rng.randint(1, min(10, beads // 12)),
                    runs=max(1, min(_log(rng, 8, 1024), int(4e7 / beads ** 2))), steps=rng.randint(25, 50))
    if kind == "train":
        c = dict(kind=kind, cvs=rng.randint(2, 40), **net, batch=_log(rng, 32, 512),
                 dropout=rng.choice([0.0, 0.1, 0.1]), labels=_log(rng, 600, 20000))
        c["steps"] = _capped_steps(rng, 4, 20, 3.0 * _mlp_flops(c) * c["batch"], 4e10)
        return c
    if kind in ("mcmc", "mcmc_system"):
        c = dict(kind=kind, cvs=rng.randint(2, 40), **net, walkers=_log(rng, 100, 4000), bins=rng.randint(40, 101))
        if kind == "mcmc_system":
            c["precision"] = rng.choice(["bf16", "bf16", "fp8"])
        c["steps"] = _capped_steps(rng, 4, 50, 0.5 * _mlp_flops(c) * c["walkers"], 1.6e11)
        return c
    lower = rng.randint(4, 40)
    return dict(kind="select", frames=_log(rng, 2000, 102400), cvs=rng.randint(2, 20), threshold=rng.uniform(1.0, 4.0),
                lower=lower, upper=lower + rng.randint(5, 20), max_selection=50)


# ---------------------------------------------------------------------------
# inputs
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _uniform(g, lo, hi, *shape, dtype=torch.float32):
    return torch.rand(*shape, generator=g, device="cuda", dtype=dtype) * (hi - lo) + lo


def _chains(walkers, beads, g, tries=24, min_dist=0.9):
    """Self-avoiding starting chains [W][N][3] grown bead by bead: unit bonds, 110 degree angles, of `tries` random
    dihedrals the first that keeps `min_dist` from every earlier bead.  Spare chains are grown for those that get
    trapped; if the spares do not suffice, free chains serve twice."""
    th = math.radians(110.0)
    want, walkers = walkers, walkers + walkers // 4 + 16
    free = torch.ones(walkers, dtype=torch.bool, device="cuda")
    x = torch.zeros(walkers, beads, 3, device="cuda")
    x[:, 1, 0] = 1.0
    x[:, 2, 0] = 1.0 - math.cos(th)
    x[:, 2, 1] = math.sin(th)
    phi = _uniform(g, -math.pi, math.pi, beads, walkers, tries)
    order = torch.arange(tries, 0, -1, device="cuda", dtype=torch.float32)
    for i in range(3, beads):
        a, b, c = x[:, i - 3], x[:, i - 2], x[:, i - 1]
        bc = torch.nn.functional.normalize(c - b, dim=-1)
        n = torch.nn.functional.normalize(torch.linalg.cross(b - a, bc), dim=-1)
        m = torch.linalg.cross(n, bc)
        p = phi[i][..., None]
        cand = (c - math.cos(th) * bc)[:, None] + math.sin(th) * (torch.cos(p) * m[:, None] + torch.sin(p) * n[:, None])
        far = (cand[:, :, None] - x[:, None, : i - 2]).square().sum(-1).amin(-1)
        # a valid candidate outranks any other; the first valid one outranks the later ones
        valid = far >= min_dist * min_dist
        best = torch.where(valid, 1e3 * order, far).argmax(-1)
        x[:, i] = cand.gather(1, best[:, None, None].expand(-1, 1, 3))[:, 0]
        free &= valid.any(-1)
    first = torch.argsort(free.logical_not().to(torch.int8), stable=True)      # free chains first, in order
    x = x[first[torch.arange(want, device="cuda") % free.sum().clamp(min=1)]]
    return (x - x.mean(1, keepdim=True)).contiguous()


def _velocities(x, g):
    return torch.randn(x.shape, generator=g, device="cuda")


def _system_params(case, seed, beads=None, cvs=None):
    return I.make_system(beads or case["beads"], cvs or case["cvs"], int(seed),
                         output_freq=max(1, min(50, case.get("steps", 1) // 2)))


def _ensemble_params(case, seed):
    return I.make_ensemble(case["models"], 2 * case["cvs"], case["layers"], case["width"], int(seed),
                           resnet=case["resnet"])


def _labels_of(case, steps):
    """(equilibration, blocks) of a labeling run: a tenth, and ten blocks."""
    return steps // 10, 10


def _label_inputs(sp, runs, seed):
    """Start, velocities, restraint centres near the start's own CVs, force constants."""
    g = _gen(seed)
    x = _chains(runs, sp.n_beads, g)
    v = _velocities(x, g)
    s0 = _torsions(x.to(F64), torch.from_numpy(sp.cv_atoms).long().cuda()[None])
    s0 = s0 + _uniform(g, -0.3, 0.3, *s0.shape, dtype=F64)
    return x, v, s0.contiguous(), _uniform(g, 50.0, 500.0, *s0.shape, dtype=F64)


def _batch_specs(case):
    return I.label_batch_jobs(case["jobs"], case["mix"], n_lo=case["beads_lo"], n_hi=case["beads_hi"],
                              cv_lo=case["cvs_lo"], cv_hi=case["cvs_hi"], n_steps=case["steps"])


def _batch_inputs(case, seed):
    """[(system parameters, x0, v0, s0, kappa)] on the host."""
    specs = _batch_specs(case)
    g = _gen(seed)
    out = [None] * len(specs)
    # shorter chains are the first beads of longer ones
    grown = _chains(len(specs), max(j["n_beads"] for j in specs), g)
    vel = _velocities(grown, g)
    off = _uniform(g, -0.3, 0.3, len(specs), max(j["n_cv"] for j in specs), dtype=F64)
    sps = [I.make_system(j["n_beads"], j["n_cv"], j["seed"] ^ int(seed)) for j in specs]
    cv = _padded_cvs(sps)
    s = (_torsions(grown.to(F64), cv) + off).cpu().numpy()
    grown, vel = grown.cpu().numpy(), vel.cpu().numpy()
    for k, (j, sp) in enumerate(zip(specs, sps)):
        N, C = sp.n_beads, sp.n_cv
        out[k] = (sp, np.ascontiguousarray(grown[k:k + 1, :N]), np.ascontiguousarray(vel[k:k + 1, :N]),
                  np.ascontiguousarray(s[k:k + 1, :C]), np.ascontiguousarray(j["kappa"][None, :]))
    return out


def _constrained_inputs(case, seed):
    g = _gen(seed)
    x = _chains(case["runs"], case["beads"], g)
    v = _velocities(x, g)
    stride = case["beads"] // case["pairs"]
    first = np.arange(case["pairs"], dtype=np.int32) * stride
    pairs = np.ascontiguousarray(np.stack([first, first + min(10, stride // 2)], axis=1).astype(np.int32))
    idx = torch.from_numpy(pairs).long().cuda()
    d0 = (x[:, idx[:, 0]] - x[:, idx[:, 1]]).to(F64).norm(dim=-1).contiguous()
    return x, v, pairs, d0


def _train_inputs(case, seed):
    g = _gen(seed)
    C = case["cvs"]
    s = _uniform(g, -math.pi, math.pi, case["labels"], C)
    # mean forces of a smooth periodic free energy, with the scatter of a finite labeling run
    amp, ph = _uniform(g, 0.5, 3.0, C), _uniform(g, -math.pi, math.pi, C)
    mf = amp * torch.sin(s + ph) + 0.5 * torch.sin(s + torch.roll(s, 1, 1))
    mf = (mf + 0.1 * torch.randn(mf.shape, generator=g, device="cuda")).contiguous()
    idx = torch.randint(0, case["labels"], (case["steps"], case["models"], case["batch"]), generator=g, device="cuda",
                        dtype=torch.int32)
    return s, mf, idx


def _mcmc_inputs(case, seed):
    g = _gen(seed)
    return _uniform(g, -math.pi, math.pi, case["walkers"], case["cvs"])


def _select_inputs(case, seed):
    """CV and deviation traces as exploration leaves them: torus walks, 100 frames a walker."""
    g = _gen(seed)
    W, C = (case["frames"] + 99) // 100, case["cvs"]
    cv = torch.cumsum(0.15 * torch.randn(W, 100, C, generator=g, device="cuda"), 1)
    cv = cv + _uniform(g, -math.pi, math.pi, W, 1, C)
    cv = torch.remainder(cv + math.pi, 2 * math.pi) - math.pi
    eps = _uniform(g, 0.0, 4.0, W * 100)
    return cv.reshape(-1, C)[: case["frames"]].contiguous(), eps[: case["frames"]].contiguous()


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("explore", "forces"):
        sp, ens, g = _system_params(case, seed), _ensemble_params(case, seed), _gen(seed)
        system = rid.System(sp)
        system.set_ensemble(ens, precision=PRECISION[case["precision"]])
        x = _chains(case["walkers"], case["beads"], g)
        W, C, N = case["walkers"], case["cvs"], case["beads"]
        st = dict(case=case, system=system, x=x)
        if kind == "explore":
            T = case["steps"] // sp.output_freq
            st.update(v=_velocities(x, g), cv=torch.zeros(W, T, C, device="cuda"), eps=torch.zeros(W, T, device="cuda"),
                      xo=torch.zeros_like(x), vo=torch.zeros_like(x))
        else:
            st.update(f=torch.zeros_like(x), s=torch.zeros(W, C, device="cuda"), eps=torch.zeros(W, device="cuda"),
                      abar=torch.zeros(W, device="cuda"), grad=torch.zeros(case["models"], W, C, device="cuda"))
        return st
    if kind == "label":
        sp = _system_params(case, seed)
        x, v, s0, kappa = _label_inputs(sp, case["runs"], seed)
        return dict(case=case, system=rid.System(sp), x=x, v=v, s0=s0, kappa=kappa,
                    out=[torch.zeros_like(s0) for _ in range(3)])
    if kind == "label_batch":
        jobs = []
        eq, blocks = _labels_of(case, case["steps"])
        for sp, x, v, s0, kappa in _batch_inputs(case, seed):
            jobs.append(dict(system=rid.System(sp), x0=x, v0=v, s0=s0, kappa=kappa, n_steps=case["steps"], n_equil=eq,
                             n_blocks=blocks, mf=np.zeros_like(s0), se=np.zeros_like(s0), std=np.zeros_like(s0)))
        return dict(case=case, jobs=jobs, server=rid.Server(4 << 30))
    if kind == "constrained":
        x, v, pairs, d0 = _constrained_inputs(case, seed)
        sp = _system_params(case, seed, cvs=2)
        return dict(case=case, system=rid.System(sp), x=x, v=v, pairs=pairs, d0=d0,
                    out=[torch.zeros_like(d0) for _ in range(3)])
    if kind == "train":
        s, mf, idx = _train_inputs(case, seed)
        ens = _ensemble_params(case, seed)
        tr = rid.Trainer(case["models"], case["cvs"], case["layers"], case["width"], ens.weights,
                         batch_size=case["batch"], resnet=case["resnet"], dropout_rate=case["dropout"],
                         dropout_seed=int(seed) + 1)
        tr.set_data(s, mf)
        return dict(case=case, trainer=tr, idx=idx, loss=torch.zeros(case["steps"], case["models"], device="cuda"),
                    w=torch.zeros(ens.weights.shape, device="cuda"))
    if kind in ("mcmc", "mcmc_system"):
        C, bins = case["cvs"], case["bins"]
        st = dict(case=case, s=_mcmc_inputs(case, seed), s_out=torch.zeros(case["walkers"], C, device="cuda"),
                  hist1=torch.zeros(C, bins, dtype=torch.uint64, device="cuda"),
                  hist2=torch.zeros(bins, bins, dtype=torch.uint64, device="cuda"),
                  pmf1=torch.zeros(C, bins, dtype=F64, device="cuda"),
                  pmf2=torch.zeros(bins, bins, dtype=F64, device="cuda"), seed=int(seed))
        ens = _ensemble_params(case, seed)
        if kind == "mcmc":
            st["w"] = torch.from_numpy(ens.weights).cuda()
        else:
            st["system"] = rid.System(I.make_system(max(24, C + 8), C, int(seed)))
            st["system"].set_ensemble(ens, precision=PRECISION[case["precision"]])
        return st
    cv, eps = _select_inputs(case, seed)
    return dict(case=case, cv=cv, eps=eps, sel=torch.zeros(case["max_selection"], dtype=torch.int32, device="cuda"))


MC_KT, MC_STEP, MC_BURN = 1.0, 0.3, 2


def run(state):
    case, st = state["case"], torch.cuda.current_stream()
    kind = case["kind"]
    if kind == "explore":
        state["system"].explore(state["x"], case["steps"], v0=state["v"], cv_out=state["cv"], eps_out=state["eps"],
                                x_out=state["xo"], v_out=state["vo"], stream=st)
        return {"cv": state["cv"], "eps": state["eps"], "x": state["xo"], "v": state["vo"]}
    if kind == "forces":
        state["system"].eval_forces(state["x"], rid.RID_BIAS_ENSEMBLE, f_out=state["f"], s_out=state["s"],
                                    eps_out=state["eps"], abar_out=state["abar"], grad_out=state["grad"], stream=st)
        return {k: state[k] for k in ("f", "s", "eps", "abar", "grad")}
    if kind == "label":
        eq, blocks = _labels_of(case, case["steps"])
        state["system"].label(state["x"], state["s0"], state["kappa"], case["steps"], eq, blocks, *state["out"],
                              v0=state["v"], stream=st)
        return dict(zip(("mf", "se", "std"), state["out"]))
    if kind == "label_batch":
        state["server"].label_batch(state["jobs"], stream=st)
        return {k: np.concatenate([j[k][0] for j in state["jobs"]]) for k in ("mf", "se", "std")}
    if kind == "constrained":
        eq, blocks = _labels_of(case, case["steps"])
        state["system"].label_constrained(state["x"], state["pairs"], state["d0"], case["steps"], eq, blocks,
                                          *state["out"], v0=state["v"], stream=st)
        return dict(zip(("mf", "se", "std"), state["out"]))
    if kind == "train":
        state["trainer"].run(state["idx"], loss_out=state["loss"], stream=st)
        w, _ = state["trainer"].weights(state["w"], stream=st)
        return {"loss": state["loss"], "w": w}
    if kind in ("mcmc", "mcmc_system"):
        o = {k: state[k] for k in ("s_out", "hist1", "hist2", "pmf1", "pmf2")}
        if kind == "mcmc":
            n = rid.mcmc(state["w"], case["models"], case["cvs"], case["layers"], case["width"], state["s"],
                         case["steps"], MC_BURN, MC_KT, MC_STEP, state["seed"], bins=case["bins"],
                         resnet=case["resnet"], stream=st, **o)
        else:
            n = state["system"].mcmc(state["s"], case["steps"], MC_BURN, MC_KT, MC_STEP, state["seed"],
                                     bins=case["bins"], stream=st, **o)
        return {**{k: v.view(torch.int64) if v.dtype == torch.uint64 else v for k, v in o.items()}, "accepted": n}
    first, clusters, threshold = rid.select(state["cv"], state["eps"], 2.0, 3.0, case["threshold"], case["lower"],
                                          case["upper"], True, case["max_selection"], selected=state["sel"], stream=st)
    return {"selected": state["sel"], "count": len(first), "clusters": clusters, "threshold": threshold}


# ---------------------------------------------------------------------------
# work
def _mlp_flops(case):
    """Forward pass and input gradient of the ensemble for one walker."""
    H, D, L = case["width"], 2 * case["cvs"], case["layers"]
    return 4.0 * case["models"] * (D * H + (L - 1) * H * H + H)


def _params(case):
    H, D, L = case["width"], 2 * case["cvs"], case["layers"]
    return case["models"] * (H * D + H + (L - 1) * (H * H + H) + H + 1)


def _chain_flops(beads):
    """Force field of one chain: 20 per non-excluded pair, and some 400 per bead for bonded terms and the integrator."""
    return 20.0 * max(0, beads - 2) * max(0, beads - 3) / 2 + 400.0 * beads


def work(case):
    kind = case["kind"]
    if kind in ("explore", "forces"):
        W, N, C = case["walkers"], case["beads"], case["cvs"]
        steps = case.get("steps", 0) + 1
        chain = 12.0 * W * N
        if kind == "explore":
            T = case["steps"] // max(1, min(50, case["steps"] // 2))
            nbytes = 4 * chain + 4.0 * W * T * (C + 1) + 4.0 * _params(case)
        else:
            nbytes = 2 * chain + 4.0 * W * (C + 2 + case["models"] * C) + 4.0 * _params(case)
        return {"bytes": nbytes, "flops": steps * W * (_mlp_flops(case) + _chain_flops(N))}
    if kind in ("label", "constrained"):
        R, N = case["runs"], case["beads"]
        C = case["cvs"] if kind == "label" else case["pairs"]
        return {"bytes": R * (24.0 * N + 8.0 * C * (5 if kind == "label" else 4)),
                "flops": float(case["steps"]) * R * _chain_flops(N)}
    if kind == "label_batch":
        lo, hi = math.log(case["beads_lo"]), math.log(case["beads_hi"])
        at = [math.exp(lo + (hi - lo) * (k + 0.5) / 64) for k in range(64)]
        C = 0.5 * (case["cvs_lo"] + case["cvs_hi"])
        return {"bytes": case["jobs"] * (24.0 * sum(at) / 64 + 40.0 * C),
                "flops": float(case["jobs"]) * case["steps"] * sum(_chain_flops(n) for n in at) / 64}
    if kind == "train":
        H, D, L = case["width"], 2 * case["cvs"], case["layers"]
        per = 10.0 * (D * H + (L - 1) * H * H) + 2.0 * (L - 1) * H * H
        return {"bytes": 8.0 * _params(case) + case["steps"] * case["models"] * case["batch"] * (8.0 * case["cvs"] + 4),
                "flops": case["steps"] * case["models"] * case["batch"] * per}
    if kind in ("mcmc", "mcmc_system"):
        W, C, b = case["walkers"], case["cvs"], case["bins"]
        return {"bytes": 4.0 * _params(case) + 8.0 * W * C + 16.0 * (C * b + b * b),
                "flops": (case["steps"] + 1) * W * 0.5 * _mlp_flops(case)}
    # a frame in four is a candidate; each is compared with about half of the leaders of the final clustering
    n, C = case["frames"], case["cvs"]
    return {"bytes": 4.0 * n * (C + 1), "flops": 0.25 * n * 0.5 * case["upper"] * 8.0 * C}


# ---------------------------------------------------------------------------
# the same quantities in 64 bits, from their definitions
def _wrap(d):
    return d - 2 * math.pi * torch.floor(d / (2 * math.pi) + 0.5)


def _torsion(p0, p1, p2, p3):
    b1, b2, b3 = p1 - p0, p2 - p1, p3 - p2
    m, n = torch.linalg.cross(b1, b2), torch.linalg.cross(b2, b3)
    phi = torch.atan2(b2.norm(dim=-1) * (b1 * n).sum(-1), (m * n).sum(-1))
    return torch.where(phi >= math.pi, phi - 2 * math.pi, phi)


def _torsions(x, cv):
    """Torsions [W][C] of x [W][N][3] for quadruples cv [W or 1][C][4]."""
    W, C = x.shape[0], cv.shape[1]
    p = x.gather(1, cv.expand(W, C, 4).reshape(W, 4 * C, 1).expand(-1, -1, 3)).view(W, C, 4, 3)
    return _torsion(p[:, :, 0], p[:, :, 1], p[:, :, 2], p[:, :, 3])


def _padded_cvs(sps):
    C = max(sp.n_cv for sp in sps)
    cv = np.tile(np.arange(4, dtype=np.int64), (len(sps), C, 1))
    for k, sp in enumerate(sps):
        cv[k, : sp.n_cv] = sp.cv_atoms
    return torch.from_numpy(cv).cuda()


def _philox(c0, c1, c2, c3, key):
    """Philox4x32-10 words (int64 tensors of 32-bit values)."""
    mask = 0xFFFFFFFF
    k0, k1 = key & mask, (key >> 32) & mask
    for _ in range(10):
        p0, p1 = 0xD2511F53 * c0, 0xCD9E8D57 * c2
        c0, c1, c2, c3 = ((p1 >> 32) & mask) ^ c1 ^ k0, p1 & mask, ((p0 >> 32) & mask) ^ c3 ^ k1, p0 & mask
        k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
    return c0, c1, c2, c3


def _normals(a, b, step, stream, key):
    """Box-Muller triples [..., 3] of counters (a, b, step, stream)."""
    a, b = torch.broadcast_tensors(a, b)
    words = _philox(a, b, torch.full_like(a, step), torch.full_like(a, stream), key)
    u = [(w.to(F64) + 0.5) * 2.0 ** -32 for w in words]
    r0, r1 = torch.sqrt(-2 * torch.log(u[0])), torch.sqrt(-2 * torch.log(u[2]))
    return torch.stack([r0 * torch.cos(2 * math.pi * u[1]), r0 * torch.sin(2 * math.pi * u[1]),
                        r1 * torch.cos(2 * math.pi * u[3])], -1)


class _Chains:
    """Force field and BAOAB steps of W chains in 64 bits; chains of unequal length are padded with frozen beads."""

    def __init__(self, sps, walkers):
        sp = sps[0]
        self.sp, N = sp, max(p.n_beads for p in sps)
        self.n = torch.tensor([p.n_beads for p in sps], device="cuda").expand(walkers if len(sps) == 1 else len(sps))
        dk, dd = np.zeros((len(sps), N - 3, 3)), np.zeros((len(sps), N - 3, 3))
        for k, p in enumerate(sps):
            dk[k, : p.n_beads - 3], dd[k, : p.n_beads - 3] = p.dihedral_k, p.dihedral_delta
        self.dk, self.dd = torch.from_numpy(dk).cuda(), torch.from_numpy(dd).cuda()
        self.keys = torch.tensor([int(p.seed) for p in sps], device="cuda").reshape(-1, 1)
        self.own = self.n[:, None] > torch.arange(N, device="cuda")          # [W][N] real beads
        i = torch.arange(N, device="cuda")
        self.apart = (i[:, None] - i[None]).abs() >= 3

    def bonded_force(self, x):
        sp = self.sp
        with torch.enable_grad():
            x = x.detach().requires_grad_(True)
            d = x[:, 1:] - x[:, :-1]
            own = self.own.to(F64)
            U = (own[:, 1:] * 0.5 * sp.bond_k * (d.norm(dim=-1) - sp.bond_r0) ** 2).sum()
            a, b = -d[:, :-1], d[:, 1:]
            th = torch.atan2(torch.linalg.cross(a, b).norm(dim=-1), (a * b).sum(-1))
            U = U + (own[:, 2:] * 0.5 * sp.angle_k * (th - sp.angle_theta0) ** 2).sum()
            phi = _torsion(x[:, :-3], x[:, 1:-2], x[:, 2:-1], x[:, 3:])[..., None]
            n = torch.arange(1, 4, device="cuda", dtype=F64)
            U = U + (own[:, 3:, None] * self.dk * (1 + torch.cos(n * phi - self.dd))).sum()
            return -torch.autograd.grad(U, x)[0]

    def lj_force(self, x):
        sp = self.sp
        rc2, s2 = float(np.float32(sp.lj_rc ** 2)), sp.lj_sigma ** 2
        f = torch.empty_like(x)
        per = max(1, int(4e7 / x.shape[1] ** 2))
        for w in range(0, x.shape[0], per):
            y, own = x[w:w + per], self.own[w:w + per]
            d = [y[:, None, :, k] - y[:, :, None, k] for k in range(3)]
            r2 = d[0] ** 2 + d[1] ** 2 + d[2] ** 2
            take = self.apart & (r2 < rc2) & own[:, None] & own[:, :, None]
            i2 = torch.where(take, 1.0 / r2, 0.0)
            s6 = (s2 * i2) ** 3
            c = 24.0 * sp.lj_eps * (2 * s6 * s6 - s6) * i2
            f[w:w + per] = torch.stack([-(c * dk).sum(-1) for dk in d], -1)
        return f

    def force(self, x):
        return (self.bonded_force(x) + self.lj_force(x)) * self.own[..., None]

    def cv_force(self, x, cv, of_s):
        """(s, sum_j F_j ds_j/dx) where F = of_s(s)."""
        with torch.enable_grad():
            x = x.detach().requires_grad_(True)
            s = _torsions(x, cv)
            F = of_s(s.detach())
            return s.detach(), torch.autograd.grad((s * F).sum(), x)[0]

    def noise(self, step, single):
        """Walker index 0 for runs that are jobs of their own, else the row."""
        W, N = self.own.shape
        bead = torch.arange(N, device="cuda").expand(W, N)
        row = torch.zeros_like(bead) if single else torch.arange(W, device="cuda")[:, None].expand(W, N)
        return _normals(bead, row, step, 0, self.keys.expand(W, N) if single else int(self.sp.seed))

    def coefficients(self):
        sp = self.sp
        c1 = math.exp(-sp.gamma * sp.dt)
        return 0.5 * sp.dt, c1, math.sqrt((1 - c1 * c1) * sp.kT / sp.mass)

    def pad(self, xs):
        """[W][N][3] from a list of chains; a padded bead sits on a far zigzag that no term reads."""
        W, N = self.own.shape
        i = torch.arange(N, device="cuda", dtype=F64)
        x = torch.stack([1e3 + i, i % 2, (i // 2) % 2], -1).expand(W, N, 3).clone()
        v = torch.zeros_like(x)
        for k, (a, b) in enumerate(xs):
            x[k, : a.shape[0]], v[k, : a.shape[0]] = a, b
        return x, v


def _exact_ensemble(case, weights):
    """s [W][C] -> (A [M][W], dA/ds [M][W][C])."""
    H, D, L = case["width"], 2 * case["cvs"], case["layers"]
    w = torch.from_numpy(np.asarray(weights)).cuda().to(F64)
    layers, o, fin = [], 0, D
    for _ in range(L):
        layers.append((w[:, o:o + H * fin].reshape(-1, H, fin), w[:, None, o + H * fin:o + H * fin + H]))
        o, fin = o + H * fin + H, H
    wo, bo = w[:, o:o + H], w[:, o + H]

    def ensemble(s, gradient=True):
        u = torch.stack([torch.cos(s), torch.sin(s)], -1).reshape(s.shape[0], D)
        h, ts = u.expand(w.shape[0], *u.shape), []
        for l, (W, b) in enumerate(layers):
            t = torch.tanh(torch.baddbmm(b, h, W.transpose(1, 2)))
            ts.append(t)
            h = t + h if case["resnet"] and l else t
        A = (h @ wo[..., None])[..., 0] + bo[:, None]
        if not gradient:
            return A, None
        g = wo[:, None].expand_as(h)
        for l in range(L - 1, -1, -1):
            back = (g * (1 - ts[l] ** 2)) @ layers[l][0]
            g = back + g if case["resnet"] and l else back
        return A, -torch.sin(s) * g[..., 0::2] + torch.cos(s) * g[..., 1::2]

    return ensemble


def _mean_force(grads, lo=2.0, hi=3.0):
    """(mean force, deviation, switched force)."""
    F = grads.mean(0)
    eps = ((grads - F) ** 2).sum(-1).mean(0).sqrt()
    between = 0.5 * (1 + torch.cos(math.pi * (eps - lo) / (hi - lo)))
    sw = torch.where(eps < lo, 1.0, torch.where(eps >= hi, 0.0, between))
    return F, eps, sw[:, None] * F


def _statistics(d, kappa, blocks):
    """mf, se, std of samples d [K][R][C]."""
    K = d.shape[0]
    which = (torch.arange(K, device="cuda") * blocks) // K
    means = torch.stack([d[which == b].mean(0) for b in range(blocks)])
    return {"mf": -kappa * d.mean(0), "se": kappa * means.std(0, unbiased=True) / math.sqrt(blocks),
            "std": kappa * d.std(0, unbiased=False)}


def _exact_explore(case, seed):
    sp, g = _system_params(case, seed), _gen(seed)
    x = _chains(case["walkers"], case["beads"], g)
    ch, x, v = _Chains([sp], case["walkers"]), x.to(F64), None
    ens = _exact_ensemble(case, _ensemble_params(case, seed).weights)
    cv = torch.from_numpy(sp.cv_atoms).long().cuda()[None]
    seen = {}

    def force(x):
        def bias(s):
            seen["A"], seen["grad"] = ens(s)
            _, seen["eps"], F = _mean_force(seen["grad"])
            return F
        f = ch.force(x)
        seen["s"], fb = ch.cv_force(x, cv, bias)
        return f + fb

    f = force(x)
    if case["kind"] == "forces":
        return {"f": f, "s": seen["s"], "eps": seen["eps"], "abar": seen["A"].mean(0), "grad": seen["grad"]}
    v = _velocities(x, g).to(F64)
    h, c1, c2 = ch.coefficients()
    cvs, devs = [], []
    for t in range(case["steps"]):
        v = v + h * f / sp.mass
        x = x + h * v
        v = c1 * v + c2 * ch.noise(t, False)
        x = x + h * v
        f = force(x)
        v = v + h * f / sp.mass
        if (t + 1) % sp.output_freq == 0:
            cvs.append(seen["s"])
            devs.append(seen["eps"])
    return {"cv": torch.stack(cvs, 1), "eps": torch.stack(devs, 1), "x": x, "v": v}


def _exact_labels(ch, x, v, cv, s0, kappa, steps, eq, blocks, single):
    h, c1, c2 = ch.coefficients()
    own, d = ch.own[..., None], []

    def force(x):
        s, fr = ch.cv_force(x, cv, lambda s: -kappa * _wrap(s - s0))
        return s, ch.force(x) + fr * own

    _, f = force(x)
    for t in range(steps):
        v = v + h * f / ch.sp.mass
        x = x + h * v
        v = (c1 * v + c2 * ch.noise(t, single)) * own
        x = x + h * v
        s, f = force(x)
        v = v + h * f / ch.sp.mass
        if t >= eq:
            d.append(_wrap(s - s0))
    return _statistics(torch.stack(d), kappa, blocks)


def _exact_label(case, seed):
    sp = _system_params(case, seed)
    x, v, s0, kappa = _label_inputs(sp, case["runs"], seed)
    cv = torch.from_numpy(sp.cv_atoms).long().cuda()[None]
    eq, blocks = _labels_of(case, case["steps"])
    return _exact_labels(_Chains([sp], case["runs"]), x.to(F64), v.to(F64), cv, s0, kappa, case["steps"], eq, blocks,
                         False)


def _exact_label_batch(case, seed):
    jobs = _batch_inputs(case, seed)
    sps = [j[0] for j in jobs]
    ch = _Chains(sps, len(sps))
    x, v = ch.pad([(torch.from_numpy(j[1][0]).cuda().to(F64), torch.from_numpy(j[2][0]).cuda().to(F64)) for j in jobs])
    cv = _padded_cvs(sps)
    s0, kappa = (torch.zeros(cv.shape[:2], dtype=F64, device="cuda") for _ in range(2))
    for k, j in enumerate(jobs):                       # a padded CV has no force constant
        s0[k, : sps[k].n_cv], kappa[k, : sps[k].n_cv] = torch.from_numpy(j[3][0]), torch.from_numpy(j[4][0])
    eq, blocks = _labels_of(case, case["steps"])
    o = _exact_labels(ch, x, v, cv, s0, kappa, case["steps"], eq, blocks, True)
    return {q: torch.cat([o[q][k, : sp.n_cv] for k, sp in enumerate(sps)]) for q in ("mf", "se", "std")}


def _exact_constrained(case, seed):
    x, v, pairs, d0 = _constrained_inputs(case, seed)
    sp = _system_params(case, seed, cvs=2)
    ch, x, v = _Chains([sp], case["runs"]), x.to(F64), v.to(F64)
    a, b = (torch.from_numpy(pairs[:, k]).long().cuda() for k in (0, 1))
    h, c1, c2 = ch.coefficients()

    def project(x, v):
        u = x[:, a] - x[:, b]
        u = u / u.norm(dim=-1, keepdim=True)
        w = 0.5 * ((v[:, a] - v[:, b]) * u).sum(-1, keepdim=True) * u
        v = v.clone()
        v[:, a] -= w
        v[:, b] += w
        return v

    def drift(x, v):
        old, x = x[:, a] - x[:, b], x + h * v
        new = x[:, a] - x[:, b]
        oo, no, nn = ((p * q).sum(-1) for p, q in ((old, old), (new, old), (new, new)))
        lam = (nn - d0 ** 2) / (2 * (no + torch.sqrt((no ** 2 - oo * (nn - d0 ** 2)).clamp(min=0))))
        move = lam[..., None] * old
        v = v.clone()
        for idx, sign in ((a, -1.0), (b, 1.0)):
            x[:, idx] += sign * move
            v[:, idx] += sign * move / h
        return x, project(x, v)

    mid, u = 0.5 * (x[:, a] + x[:, b]), x[:, a] - x[:, b]
    u = 0.5 * d0[..., None] * u / u.norm(dim=-1, keepdim=True)
    x[:, a], x[:, b] = mid + u, mid - u
    v, f, F = project(x, v), ch.force(x), []
    eq, blocks = _labels_of(case, case["steps"])
    for t in range(case["steps"]):
        v = project(x, v + h * f / sp.mass)
        x, v = drift(x, v)
        v = project(x, c1 * v + c2 * ch.noise(t, False))
        x, v = drift(x, v)
        f = ch.force(x)
        v = project(x, v + h * f / sp.mass)
        if t >= eq:
            F.append(-0.5 * ((f[:, a] - f[:, b]) * (x[:, a] - x[:, b])).sum(-1) / d0 - 2 * sp.kT / d0)
    return _statistics(-torch.stack(F), torch.ones_like(d0), blocks)


def _exact_train(case, seed):
    s_all, mf_all, idx = _train_inputs(case, seed)
    M, B, C, H, L = (case[k] for k in ("models", "batch", "cvs", "width", "layers"))
    D, p = 2 * C, case["dropout"]
    w = torch.from_numpy(_ensemble_params(case, seed).weights).cuda().to(F64)
    m, v2, losses = torch.zeros_like(w), torch.zeros_like(w), []
    blocks = (H + 3) // 4
    ids = torch.arange(blocks, device="cuda")
    for t in range(case["steps"]):
        rows = idx[t].long()
        s, mf = s_all[rows].to(F64), mf_all[rows].to(F64)                      # [M][B][C]
        q = []
        for l in range(L):
            if not p:
                q.append(torch.ones((), dtype=F64, device="cuda"))
                continue
            c0 = (ids + blocks * l)[None, None] + (blocks * L * torch.arange(M, device="cuda"))[:, None, None]
            c1 = torch.arange(B, device="cuda")[None, :, None]
            c0, c1 = torch.broadcast_tensors(c0, c1)
            words = torch.stack(_philox(c0, c1, torch.full_like(c0, t), torch.full_like(c0, 4), int(seed) + 1), -1)
            q.append((words.reshape(M, B, -1)[..., :H] >= int(p * 2 ** 32)).to(F64) / (1 - p))
        with torch.enable_grad():
            w.requires_grad_(True)
            s.requires_grad_(True)
            h, o, fin = torch.stack([torch.cos(s), torch.sin(s)], -1).reshape(M, B, D), 0, D
            for l in range(L):
                W, b = w[:, o:o + H * fin].reshape(M, H, fin), w[:, None, o + H * fin:o + H * fin + H]
                z = q[l] * torch.tanh(torch.baddbmm(b, h, W.transpose(1, 2)))
                h = z + h if case["resnet"] and l else z
                o, fin = o + H * fin + H, H
            A = h @ w[:, o:o + H, None]
            dA = torch.autograd.grad(A.sum(), s, create_graph=True)[0]
            loss = ((dA - mf) ** 2).mean((1, 2))
            gw = torch.autograd.grad(loss.sum(), w)[0]
        losses.append(loss.detach())
        w = w.detach()
        m, v2 = 0.9 * m + 0.1 * gw, 0.999 * v2 + 0.001 * gw * gw
        lr = 8e-4 * 0.96 ** (t / 120)
        w = w - lr * (m / (1 - 0.9 ** (t + 1))) / ((v2 / (1 - 0.999 ** (t + 1))).sqrt() + 1e-8)
    return {"loss": torch.stack(losses), "w": w}


def _exact_mcmc(case, seed):
    s, C, bins = _mcmc_inputs(case, seed).to(F64), case["cvs"], case["bins"]
    ens = _exact_ensemble(case, _ensemble_params(case, seed).weights)
    row, col = torch.arange(case["walkers"], device="cuda")[:, None], torch.arange(C, device="cuda")[None]
    key = int(seed)
    A = ens(s, False)[0].mean(0)
    h1, h2 = torch.zeros(C * bins, dtype=F64, device="cuda"), torch.zeros(bins * bins, dtype=F64, device="cuda")
    accepted = 0
    for t in range(case["steps"]):
        xi = _normals((col // 3).expand(len(s), -1), row, t, 2, key)
        new = _wrap(s + float(np.float32(MC_STEP)) * xi.gather(-1, (col % 3).expand(len(s), -1)[..., None])[..., 0])
        An = ens(new, False)[0].mean(0)
        zero = torch.zeros(len(s), dtype=torch.int64, device="cuda")
        u = (_philox(zero, row[:, 0], zero + t, zero + 3, key)[0].to(F64) + 0.5) * 2.0 ** -32
        ok = MC_KT * torch.log(u) + (An - A) < 0
        s, A = torch.where(ok[:, None], new, s), torch.where(ok, An, A)
        accepted += int(ok.sum())
        if t >= MC_BURN:
            b = ((s + math.pi) / (2 * math.pi) * bins).floor().long().clamp(0, bins - 1)
            h1 += torch.bincount((col * bins + b).reshape(-1), minlength=C * bins)
            h2 += torch.bincount(b[:, 0] * bins + b[:, 1], minlength=bins * bins)

    def pmf(h):
        f = -MC_KT * torch.log(h / h.sum(-1, keepdim=True))
        return f - f.amin(-1, keepdim=True)

    return {"s_out": s, "hist1": h1.reshape(C, bins).long(), "hist2": h2.reshape(bins, bins).long(),
            "pmf1": pmf(h1.reshape(C, bins)), "pmf2": pmf(h2[None]).reshape(bins, bins), "accepted": accepted}


def exact(case, seed):
    """What run() returns in 64 bits.  None where a decision in lower precision has no such value (the reduced
    precision Metropolis walk; the selection, whose distances are compared in FP32 by definition), and for runs whose
    64-bit trajectory would take too long."""
    kind = case["kind"]
    w = work(case)["flops"]
    with torch.no_grad():
        if kind in ("explore", "forces"):
            pairs = (case.get("steps", 0) + 1.0) * case["walkers"] * case["beads"] ** 2
            return None if w > EXACT_FLOPS or pairs > EXACT_PAIRS else _exact_explore(case, seed)
        if kind == "label":
            return _exact_label(case, seed)
        if kind == "label_batch":
            return _exact_label_batch(case, seed)
        if kind == "constrained":
            return _exact_constrained(case, seed)
        if kind == "train":
            return _exact_train(case, seed)
        if kind == "mcmc":
            return _exact_mcmc(case, seed)
    return None
