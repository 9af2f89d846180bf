"""Performance cases of the LoRDO optimizer hot path.

A case is one call sequence of a training program that uses ``paper_2602_04396_b200.lordo.Lordo``:

* ``step``     one ``inner_step`` on gradients that lie in HBM
* ``host``     one ``inner_step_host`` on gradients that lie in pinned host memory
* ``refresh``  one ``refresh_subspace``: of the Local rule, before the first step of a round, or of the Global
               rule, from the pseudo-gradient of the synchronisation that a restored checkpoint stopped behind
* ``round``    ``H`` inner steps and ``outer_step``; with the refresh of the variant's rule where ``check`` is set

``mats`` lists the weight matrices as ``<m>x<n>r<rank>``, with ``R`` behind the rank for a matrix that is
projected from the right and ``*<count>`` for repetitions.
"""
from __future__ import annotations

import re
from typing import Dict, List, Tuple

import torch

from paper_2602_04396_b200 import lordo, synth

LR, BETA1, BETA2 = 0.004, 0.999, 0.999  # the hyper-parameters of the benchmark
LR_ROUND = 0.02  # a round's pseudo-gradient then stands well above the storage rounding of bf16 weights
OMEGA = {lordo.QHM_NONE: 1.0, lordo.QHM_LOW: 0.94, lordo.QHM_FULL: 0.97}
NO_SYNC = 1 << 30  # H of the cases that take single steps: the synchronisation is not part of them

LAYER_768 = "768x768r128*4,768x3072r128*2,3072x768r128"      # one decoder layer of the 125M-shaped stack
LAYER_2048 = "2048x2048r256*4,2048x5632r256*2,5632x2048r256"  # one decoder layer of the 1B-shaped stack
LAYERS_2048 = "2048x2048r256*8,2048x5632r256*4,5632x2048r256*2"  # two of them


def listed() -> List[dict]:
    base = dict(variant="global", form=lordo.QHM_FULL, ef=True, dtype="bf16", check=0, q=0, H=2, grad="lowrank", rho=0.5)
    local = dict(base, variant="local", form=lordo.QHM_LOW)
    return [
        # one small fp32 matrix in the binding's default mode: a toy model or a parity run, all latency
        dict(base, name="step_256_f32_check", kind="step", mats="256x256r16", K=2, dtype="f32", check=1, grad="gauss", rho=1.0),
        # one layer's matrix with fp32 storage and tensor-core contractions
        dict(base, name="step_2048_f32", kind="step", mats="2048x2048r128", K=4, dtype="f32", rho=1.0),
        # every piece of the path in fp32 arithmetic, ragged sizes: a parity run or an fp32 training run
        dict(base, name="round_ragged_f32_check", kind="round", mats="1000x1336r72,520x392r136,200x136r24", K=3, dtype="f32", check=1, q=1, rho=1.0),
        # an ordinary small step: one decoder layer of the 125M-shaped stack
        dict(local, name="step_layer768_bf16", kind="step", mats=LAYER_768, K=8),
        # the large step: two decoder layers of the 1B-shaped stack (what a rank that holds a slice of the model runs)
        dict(base, name="step_layers2048_bf16", kind="step", mats=LAYERS_2048, K=8, rho=0.1),
        # sizes that fill no tile, some projected from the right: embeddings, heads, adapters
        dict(base, name="step_ragged_bf16", kind="step", mats="1000x1336r72,2056x520r200R,504x3000r136,1032x704r96R,136x2088r64", K=3, grad="student", rho=1.0),
        # the largest rank
        dict(local, name="step_r512_bf16", kind="step", mats="4096x11008r512", K=4, grad="student", rho=1.0),
        # subspace refresh of a decoder layer, one basis per worker
        dict(local, name="refresh_layer768_bf16", kind="refresh", mats=LAYER_768, K=8),
        # the refresh stress: large rank, two subspace iterations, sixteen workers
        dict(local, name="refresh_r512_bf16", kind="refresh", mats="4096x11008r512", K=16, q=2, grad="student", rho=1.0),
        # the same of the Global rule, one basis per matrix, a layer of the 1B-shaped stack
        dict(base, name="refresh_layer2048_global", kind="refresh", mats=LAYER_2048, K=8),
        # a round of a decoder layer of the 1B-shaped stack, short so that the synchronisation counts
        dict(base, name="round_layer2048_bf16", kind="round", mats=LAYER_2048, K=8, rho=0.1),
        # gradients that arrive in host memory
        dict(base, name="host_layer768_bf16", kind="host", mats=LAYER_768, K=4),
    ]


def draw(rng) -> dict:
    """One more case: kind, number and shapes of the matrices, rank, workers, storage and options drawn."""
    kind = rng.choices(["step", "refresh", "round", "host"], [5, 2, 2, 1])[0]
    dtype, check = rng.choices([("bf16", 0), ("f32", 0), ("f32", 1)], [6, 2, 2])[0]
    variant = "global" if kind == "round" and not check else rng.choice(["global", "local"])
    budget = 4e7 if check else 3e8 if kind != "host" else 5e7  # weight-replicas
    K = rng.choice([1, 2, 3, 4, 8, 16])
    mats, weights = [], 0

    def size():
        return max(64, int(2.0 ** rng.uniform(6.0, 12.6)) // 8 * 8)

    for _ in range(rng.randint(1, 7)):
        m, n = size(), size()
        most = min(m, n, 512 if dtype == "bf16" else 256)
        r = max(8, min(most, int(min(m, n) * 2.0 ** rng.uniform(-4.0, -1.0)) // 8 * 8))
        if mats and (weights + m * n) * K > budget:
            continue
        while m * n * K > budget and K > 1:
            K -= 1
        right = dtype == "bf16" and m > n and rng.random() < 0.3
        mats.append(f"{m}x{n}r{r}{'R' if right else ''}")
        weights += m * n
    grad = rng.choice(["gauss", "lowrank", "student"])
    if kind == "refresh" and grad == "lowrank" and dtype == "bf16":
        q = 0  # more iterations only amplify the rounding of the directions behind the signal
    else:
        q = rng.choice([0, 0, 1, 2])
    return dict(kind=kind, mats=",".join(mats), K=K, variant=variant, form=rng.choice([lordo.QHM_NONE, lordo.QHM_LOW, lordo.QHM_FULL]),
                ef=rng.random() < 0.85, dtype=dtype, check=check, q=q, H=rng.choice([1, 2, 4]), grad=grad,
                rho=rng.choice([0.1, 0.5, 1.0]))


def _mats(text: str) -> Tuple[List[Tuple[int, int, int]], Tuple[int, ...]]:
    mats, sides = [], []
    for part in text.split(","):
        m, n, r, right, count = re.fullmatch(r"(\d+)x(\d+)r(\d+)(R?)(?:\*(\d+))?", part).groups()
        mats += [(int(m), int(n), int(r))] * int(count or 1)
        sides += [1 if right else 0] * int(count or 1)
    return mats, tuple(sides)


def _workload(case: dict) -> synth.Workload:
    mats, sides = _mats(case["mats"])
    dt = case["dtype"]
    return synth.Workload("case", tuple(mats), K=case["K"], H=case["H"], rounds=1, w_dtype=dt, g_dtype=dt, e_dtype=dt, grad=case["grad"],
                          power_iters=case["q"], clip_rho=case["rho"], sides=sides)


def prepare(case: dict, seed: int) -> Dict:
    """An optimizer one step into its run (at the start of one before a round), and the next gradients.

    Adam's epsilon is set to the size of a typical clipped gradient entry: with 1e-8 the first steps' update is
    the sign of its low-rank gradient, and entries below the rounding of their operands would flip it."""
    wl = _workload(case)
    kind, form = case["kind"], case["form"]
    H = {"step": NO_SYNC, "host": NO_SYNC, "refresh": 1, "round": case["H"]}[kind]
    dt = synth.torch_dtype(wl.w_dtype)
    opt = lordo.Lordo(wl.mats, wl.K, H, synth.init_weights_device(wl, seed), g_dtype=dt, e_dtype=dt,
                      variant=lordo.LOCAL if case["variant"] == "local" else lordo.GLOBAL, error_feedback=case["ef"], beta2=BETA2,
                      eps=wl.clip_rho / wl.weights ** 0.5, clip_rho=wl.clip_rho, outer=lordo.OUTER_NESTEROV, outer_lr=0.8, outer_momentum=0.9,
                      power_iters=wl.power_iters, seed=seed, check_mode=case["check"], sides=wl.sides)
    state = dict(opt=opt, kind=kind, form=form, H=H, with_refresh=bool(case["check"]))
    G = synth.gradients_device(wl, seed, 0, 0)
    if opt.variant == lordo.LOCAL:
        opt.refresh_subspace(G, BETA1)
    if kind != "round":
        opt.inner_step(G, LR, BETA1, OMEGA[form], form)
    if kind == "refresh":
        opt.outer_step()
    if kind == "refresh" and opt.variant == lordo.GLOBAL:
        # a pseudo-gradient of the gradients' kind, of the size that lr gives a round
        for d, g in zip(opt.Delta, synth.gradients_device(wl, seed, 1, 0)):
            d.copy_(g.float().mean(0) * LR)
        state["counters"] = opt.counters()
    else:
        # the coming gradients, in buffers of their own; a round alternates between two sets
        state["G"] = [synth.gradients_device(wl, seed, 1, h) for h in range(2 if kind == "round" else 1)]
    if kind == "host":
        state["host"] = [torch.empty(g.shape, dtype=g.dtype, pin_memory=True).copy_(g) for g in state["G"][0]]
        state["clip"] = torch.empty(wl.K, dtype=torch.float32, pin_memory=True)
        for g in state["G"][0]:
            g.zero_()  # from here on the staging buffers of the copies
    torch.cuda.synchronize()
    return state


def run(state: Dict):
    opt, kind, form = state["opt"], state["kind"], state["form"]
    omega = OMEGA[form]
    if kind == "step":
        opt.inner_step(state["G"][0], LR, BETA1, omega, form)
        return opt.W, opt.E, opt.u, opt.v
    if kind == "host":
        opt.inner_step_host(state["host"], state["G"][0], LR, BETA1, omega, form, state["clip"])
        return opt.W, opt.E, opt.u, opt.v, state["clip"]
    if kind == "refresh":
        if opt.variant == lordo.LOCAL:
            opt.refresh_subspace(state["G"][0], BETA1)
        else:
            opt.set_counters(state["counters"])  # resume behind the synchronisation (host work only)
            opt.refresh_subspace(None, BETA1)
        return opt.P, opt.u, opt.v
    for h in range(state["H"]):
        if state["with_refresh"] and opt.variant == lordo.LOCAL and h == 0:
            opt.refresh_subspace(state["G"][0], BETA1)
        opt.inner_step(state["G"][h & 1], LR_ROUND, BETA1, omega, form)
    opt.outer_step()
    if state["with_refresh"] and opt.variant == lordo.GLOBAL:
        opt.refresh_subspace(None, BETA1)
    return opt.W, opt.E, opt.P, opt.u, opt.v, opt.X0, opt.B, opt.Delta


def work(case: dict) -> Dict[str, float]:
    """What a pass cannot do without: every tensor it works on read once and, where it changes, written once;
    the contractions of the step (projection, error feedback, back-projection) and of the refresh (sketch
    products, orthonormalisation, rotation)."""
    mats, sides = _mats(case["mats"])
    K, H, q = case["K"], case["H"], case["q"]
    b = 2 if case["dtype"] == "bf16" else 4
    local = case["variant"] == "local"
    steps = {"step": 1, "host": 1, "refresh": 0, "round": H}[case["kind"]]
    nbytes = flops = 0.0
    for (m, n, r), side in zip(mats, sides):
        pm, ln = (n, m) if side else (m, n)
        basis = (K if local else 1) * pm * r * 4.0
        states = 2 * K * r * ln * 4.0  # u and v
        stream = K * m * n * b * 1.0
        nbytes += steps * (stream * (3 + (2 if case["ef"] else 0)) + basis + 2 * states)
        flops += steps * (3 if case["ef"] else 2) * 2.0 * K * m * n * r
        if case["kind"] == "round":  # W in and out, X0 and B in and out, Delta out, u and v in and out
            nbytes += 2 * stream + 5 * m * n * 4.0 + 2 * states
        if case["kind"] == "refresh" or (case["kind"] == "round" and case["check"]):
            nbytes += (stream * (2 if case["ef"] else 1) if local else m * n * 4.0) + 2 * basis + 2 * states
            signals = K if local else 1
            flops += signals * 2.0 * m * n * r * (1 + 2 * q)
            flops += signals * 2.0 * r * r * (pm * (1 + q) + ln * q)  # orthonormalisation of tall factors (Gram half and product)
            flops += signals * 2.0 * pm * r * r + 2 * 2.0 * K * r * r * ln  # Rot and the rotated moments
    return {"bytes": nbytes, "flops": flops}


def tolerance(case: dict) -> Dict[str, float]:
    """About four times what the rows of the matrices in another order (hence every sum over them) change."""
    f32, check = case["dtype"] == "f32", case["check"]
    if case["kind"] == "refresh":  # right-hand sides rounded to bf16, noise directions without a gap: 9e-3 seen (fp32: 3e-4, 6e-6)
        return {"rel": 3e-2, "max": 0.4} if not f32 else {"rel": 3e-4, "max": 1e-2} if check else {"rel": 1e-3, "max": 3e-2}
    if case["kind"] == "round":    # pseudo-gradients of rounded weights: 4e-3 seen (fp32: 2e-3; check mode with its refresh: 4e-5)
        return {"rel": 1.5e-2, "max": 0.9} if not f32 else {"rel": 3e-4, "max": 1e-2} if check else {"rel": 8e-3, "max": 0.1}
    if f32:                        # 2e-7 seen in check mode, 3e-4 with bf16 operands
        return {"rel": 1e-6, "max": 1e-5} if check else {"rel": 1.5e-3, "max": 0.05}
    return {"rel": 1e-2, "max": 0.1}  # 3e-3 and 0.02 seen
