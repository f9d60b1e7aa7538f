"""Performance cases of the simulated-bifurcation (SB) track solver: what a
user's program has the library do, through its public entry points, over the
range of its workloads (one replica of a small event to the 10,000-track
pile-up event and batches of uneven events).

A case is a dict of plain values:
  kind      what the program does with the context (below)
  variant   "asb", "bsb" or "dsb"
  tracks    tracks of the event; with events > 1 the events have log-uniform
            track counts in [50, tracks]
  noise     noise hits per true hit
  cuts      the name of a cut preset of the package's workloads module
  events    events in the context
  replicas  replicas R (any number: 1 for the plain form, 50 for the paper's shots)
  prec      "fp32" or "bf16" couplings
  factor    whether the program sets the shared-hit factor (sb_set_factor)
  steps     SB steps of one pass
  dt, c0    time step; c0 in units of each event's automatic value
  every     "trace": steps between energy readouts; "backward": steps between checkpoints

Kinds:
  run       a whole run from the Philox start over the full ramp, then the
            readout (energies of all replicas, best energy, replica, selection)
            and the final state
  trace     the same with an energy readout every few steps (the energy traces)
  advance   resume from a checkpoint in mid-run: set the state, advance, get the state
  readout   energies of all replicas and the best selection of a given state
  backward  loss and gradients of one training step of the schedule (sb_backward)
  solve     a new event from its hits to its tracks: build the QUBO, create the
            context, set the factor, run, read out, assemble the tracks
"""
import math

import numpy as np
import torch

import paper_2402_14718_gb300 as sb
from paper_2402_14718_gb300 import workloads

JPREC = {"fp32": sb.SB_J_FP32, "bf16": sb.SB_J_BF16}


def listed():
    def case(name, kind, variant, tracks, cuts, replicas, steps, prec="bf16", factor=False,
             events=1, noise=0.1, dt=0.5, c0=1.0, every=0):
        return dict(name=name, kind=kind, variant=variant, tracks=tracks, noise=noise, cuts=cuts,
                    events=events, replicas=replicas, prec=prec, factor=factor, steps=steps,
                    dt=dt, c0=c0, every=every)

    return [
        # the plain single-instance form on a 100-track event (one replica, FP32
        # couplings, 2000 steps): the smallest solve, all latency and launches
        case("run_event100_bsb_r1", "run", "bsb", 100, "CUTS_S8", 1, 2000, prec="fp32"),
        # one replica on a dense 1000-track event: the plain form that
        # time-to-target compares the batched form with
        case("run_event1000_bsb_r1", "run", "bsb", 1000, "CUTS_S2_35", 1, 1000, prec="fp32"),
        # energy trace of the paper's 50 shots at its second QUBO size (N ~ 10k),
        # a0 = dt = 1, readout every 20 steps; 50 replicas are no multiple of 4
        case("trace_10k_bsb_r50", "trace", "bsb", 1064, "CUTS_DENSE", 50, 400, dt=1.0, every=20),
        # 50 shots of dSB at the paper's third QUBO size (N ~ 67k)
        case("run_67k_dsb_r50", "run", "dsb", 4133, "CUTS_DENSE", 50, 300, dt=1.0),
        # the replica-parallel bSB workload (1000 tracks, 256 replicas) resumed
        # from a checkpoint, with the shared-hit factor
        case("advance_event1000_bsb_r256", "advance", "bsb", 1000, "CUTS_S2_35", 256, 32,
             factor=True),
        # aSB on a 500-track event with FP32 couplings, no factor (a QUBO that the
        # caller did not build from hits has none); without a wall the quartic
        # force wants a small time step
        case("advance_event500_asb_r128", "advance", "asb", 500, "CUTS_S2_8", 128, 32,
             prec="fp32", dt=0.1),
        # bSB on the 10,000-track pile-up event resumed from a checkpoint: the
        # largest state that gathers FP32 positions
        case("advance_event10k_bsb_r128", "advance", "bsb", 10000, "CUTS_DENSE", 128, 16,
             factor=True, noise=0.2),
        # 64 uneven events (50 to 2000 tracks each) in one context, dSB, 64
        # replicas: the throughput workload, state well above the L2
        case("run_batch64_dsb_r64", "run", "dsb", 2000, "CUTS_S1_6", 64, 500, factor=True,
             events=64),
        # the pile-up event, dSB, 128 replicas, whole run
        case("run_event10k_dsb_r128", "run", "dsb", 10000, "CUTS_DENSE", 128, 200, factor=True,
             noise=0.2),
        # FP64 readout of a 256-replica state (checkpoints of time-to-target)
        case("readout_event1000_r256", "readout", "bsb", 1000, "CUTS_S2_35", 256, 0),
        # one gradient step of schedule learning on the adjoint workload, over a
        # horizon of 40 steps (over longer ones the gradient is ill-conditioned)
        case("backward_event500_r32", "backward", "bsb", 500, "CUTS_S2_8", 32, 40, prec="fp32",
             every=16),
        # a new 500-track event, hits to tracks
        case("solve_event500_dsb_r64", "solve", "dsb", 500, "CUTS_S2_8", 64, 500, factor=True),
    ]


def _rows(tracks, cuts):
    """About how many triplets an event of this size has (interpolated in the
    logarithm over measured sizes); only sizes of drawn cases and byte counts
    come from it."""
    table = {"CUTS_S8": ((20, 60), (100, 1721), (200, 9000)),
             "CUTS_S2_35": ((100, 950), (300, 4200), (1000, 39165)),
             "CUTS_S2_8": ((100, 1000), (500, 10878), (800, 30000)),
             "CUTS_S1_6": ((50, 406), (200, 1900), (500, 6300), (1000, 20000), (2000, 91504)),
             "CUTS_DENSE": ((95, 779), (1064, 10214), (4133, 67445), (5406, 109775),
                            (10000, 472812))}[cuts]
    lt = math.log(tracks)
    for (t0, n0), (t1, n1) in zip(table, table[1:]):
        if tracks <= t1 or (t1, n1) == table[-1]:
            f = (lt - math.log(t0)) / (math.log(t1) - math.log(t0))
            return math.exp(math.log(n0) + f * (math.log(n1) - math.log(n0)))


def _nnz_per_row(n, cuts):
    """About how many couplings a row of such an event has."""
    top = {"CUTS_S8": 14.4, "CUTS_S2_35": 41.8, "CUTS_S2_8": 20.8, "CUTS_S1_6": 40.0,
           "CUTS_DENSE": 44.9}[cuts]
    at = {"CUTS_S8": 1721, "CUTS_S2_35": 39165, "CUTS_S2_8": 10878, "CUTS_S1_6": 91504,
          "CUTS_DENSE": 472812}[cuts]
    return max(2.0, top * (n / at) ** 0.6)


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["run", "run", "run", "trace", "advance", "advance", "advance", "readout",
                       "backward", "solve"])
    cuts = rng.choice(["CUTS_S8", "CUTS_S2_35", "CUTS_S2_8", "CUTS_S1_6", "CUTS_DENSE",
                       "CUTS_DENSE"])
    span = {"CUTS_S8": (30, 150), "CUTS_S2_35": (100, 1000), "CUTS_S2_8": (100, 700),
            "CUTS_S1_6": (60, 2000), "CUTS_DENSE": (100, 8000)}[cuts]
    if kind in ("backward", "solve"):
        cuts, span = "CUTS_S2_8", (100, 600)
    tracks = _log_uniform(rng, *span)
    n = _rows(tracks, cuts)
    events = 1
    if cuts == "CUTS_S1_6" and kind in ("run", "advance"):
        events = _log_uniform(rng, 2, 40)
        n = events * _rows(math.sqrt(50 * tracks), cuts) * 1.5
    # replicas: one (the plain form), the common counts, and any number
    most = max(2, min(512, int(4e7 / n)))
    pick = rng.random()
    if pick < 0.2:
        replicas = 1
    elif pick < 0.7:
        replicas = rng.choice([r for r in (8, 16, 32, 50, 64, 96, 128, 256, 512) if r <= most] or
                              [most])
    else:
        replicas = _log_uniform(rng, 2, most)
    if kind == "backward":
        replicas = min(replicas, 64)
    variant = "bsb" if kind in ("backward", "readout") else rng.choice(["bsb", "bsb", "dsb", "dsb",
                                                                        "asb"])
    # steps of one pass: at most about 1.5e9 spin-updates
    lo, hi = {"run": (50, 2000), "trace": (100, 400), "advance": (8, 40), "readout": (0, 0),
              "backward": (16, 48), "solve": (50, 600)}[kind]
    steps = 0 if hi == 0 else max(lo // 4, min(_log_uniform(rng, lo, hi),
                                                   int(1.5e9 / (n * replicas))))
    return dict(kind=kind, variant=variant, tracks=tracks,
                noise=rng.choice([0.1, 0.2]), cuts=cuts, events=events, replicas=replicas,
                prec=rng.choice(["bf16", "bf16", "fp32"]),
                factor=kind not in ("backward", "readout") and rng.random() < 0.6, steps=steps,
                dt=rng.choice([0.5, 0.5, 1.0]) if variant != "asb" else 0.1,
                c0=rng.choice([1.0, 2.0]) if variant != "asb" else 1.0,
                every={"trace": 20, "backward": rng.choice([8, 16, 64])}.get(kind, 0))


# ---------------------------------------------------------------- inputs
def _event(case, e):
    """Event e of the case: the library's synthetic event generator. The events
    belong to the case, as those of the named workloads do, so that the arrays of
    every seed have the same shapes; a seed sets the weight of the bias, the
    replicas' starts and the states."""
    tracks = case["tracks"]
    if case["events"] > 1:
        u = np.random.default_rng((tracks, e)).uniform(math.log(50), math.log(tracks))
        tracks = int(round(math.exp(u)))
    return sb.sb_event_generate(1000003 + 101 * case["tracks"] + e,
                                sb.event_params(n_tracks=tracks, noise_frac=case["noise"]))


def _build_params(case, seed):
    cuts = dict(getattr(workloads, case["cuts"]))
    cuts["w_q"] = float(np.random.default_rng((seed, 17)).uniform(0.7, 1.3))
    return sb.build_params(**cuts)


def _qubos(case, seed):
    out = []
    for e in range(case["events"]):
        q = sb.sb_qubo_build_device(_event(case, e), _build_params(case, seed))[0]
        if q.n > 0:
            out.append(q)
    return out


def _set_factor(ctx, qs):
    """The shared-hit factor of the context's QUBOs, hit ids offset per event."""
    off, members, couple, w = 0, [], None, None
    for q in qs:
        m, couple, w, n_ids = sb.sb_qubo_factor(q)
        members.append(np.where(m >= 0, m + off, -1).astype(np.int32))
        off += n_ids
    sb.sb_set_factor(ctx, off, np.concatenate(members), couple, w)


def _context(case, qs):
    if len(qs) == 1:
        q = qs[0]
        ctx = sb.sb_create(q.n, q.rowptr, q.col, q.val, q.lin, JPREC[case["prec"]])
    else:
        ctx = sb.sb_create_batch([(q.rowptr, q.col, q.val, q.lin) for q in qs],
                                 JPREC[case["prec"]])
    if case["factor"]:
        _set_factor(ctx, qs)
    return ctx


def _state(case, seed, n):
    """A state as the middle of a run has it: a share of the spins on the wall
    (x = +-1, y = 0), the others inside with momenta of similar size."""
    g = torch.Generator(device="cuda").manual_seed(7 * seed + 3)
    shape = (n, case["replicas"])

    def u():
        return torch.rand(shape, generator=g, device="cuda", dtype=torch.float32)

    x = 2.0 * u() - 1.0
    y = 0.6 * (u() - 0.5)
    if case["variant"] != "asb":
        wall = u() < 0.45
        x = torch.where(wall, torch.where(x >= 0, 1.0, -1.0), x)
        y = torch.where(wall, 0.0, y)
    return x.contiguous(), y.contiguous()


def _ramp(case):
    """The part of the linear ramp that the pass covers (device FP32)."""
    k, s = torch.arange(case["steps"], dtype=torch.float64), max(case["steps"], 1)
    if case["kind"] == "advance":
        a = 0.3 + 0.4 * k / s       # the middle of the ramp
    elif case["kind"] == "backward":
        a = 0.5 * k / max(s - 1, 1)  # a horizon that ends in mid-bifurcation
    else:
        a = k / max(s - 1, 1)
    return a.to(torch.float32).cuda().contiguous()


def prepare(case, seed):
    s = {"case": case, "seed": seed}
    if case["kind"] == "solve":
        s["event"] = _event(case, 0)
        s["params"] = _build_params(case, seed)
        return s
    qs = _qubos(case, seed)
    ctx = s["ctx"] = _context(case, qs)
    n, E, R = ctx.n, len(qs), case["replicas"]
    if case["kind"] in ("advance", "readout"):
        s["x"], s["y"] = _state(case, seed, n)
    if case["kind"] in ("run", "trace", "advance"):
        s["x_out"], s["y_out"] = (torch.empty((n, R), device="cuda") for _ in range(2))
    if case["kind"] in ("advance", "trace", "backward"):
        s["ramp"] = _ramp(case)
    if case["kind"] in ("run", "trace", "readout"):
        s["E"] = torch.empty((E, R), dtype=torch.float64, device="cuda")
        s["best_E"] = torch.empty(E, dtype=torch.float64, device="cuda")
        s["best_r"] = torch.empty(E, dtype=torch.int32, device="cuda")
        s["T"] = torch.empty(n, dtype=torch.uint8, device="cuda")
    if case["kind"] == "trace":
        s["Es"] = torch.empty((-(-case["steps"] // case["every"]), E, R), dtype=torch.float64,
                              device="cuda")
    if case["kind"] == "readout":
        sb.sb_set_state(ctx, s["x"], s["y"])
    if case["kind"] == "backward":
        q = qs[0]
        sb.sb_set_weights(ctx, q.cls, q.quality, 1.0, 1.0)
        s["c0_abs"] = case["c0"] * sb.sb_info(ctx)["c0_auto"]
        s["grad"] = torch.zeros(case["steps"], dtype=torch.float64, device="cuda")
    return s


# ---------------------------------------------------------------- one pass
def _readout(s):
    sb.sb_readout_device(s["ctx"], s["E"], s["best_E"], s["best_r"], s["T"])
    return [s["E"], s["best_E"], s["best_r"], s["T"]]


def _get_state(s):
    # the C entry point with on_device = 1 (the Python function copies to the host)
    sb._lib.check(sb.lib.sb_get_state(s["ctx"].handle, s["x_out"].data_ptr(),
                                      s["y_out"].data_ptr(), 1))
    return [s["x_out"], s["y_out"]]


def run(s):
    case = s["case"]
    variant, R, steps, dt, c0 = (case[k] for k in ("variant", "replicas", "steps", "dt", "c0"))
    if case["kind"] == "run":
        sb.sb_run(s["ctx"], variant, 1.0, -c0, dt, steps, R, s["seed"] + 1)
        return _readout(s) + _get_state(s)
    if case["kind"] == "trace":
        sb.sb_run(s["ctx"], variant, 1.0, -c0, dt, 0, R, s["seed"] + 1)
        for i, k in enumerate(range(0, steps, case["every"])):
            m = min(case["every"], steps - k)
            sb.sb_advance(s["ctx"], variant, 1.0, -c0, dt, m, s["ramp"][k:k + m])
            sb.sb_readout_device(s["ctx"], s["Es"][i])
        return [s["Es"]] + _readout(s) + _get_state(s)
    if case["kind"] == "advance":
        sb.sb_set_state(s["ctx"], s["x"], s["y"])
        sb.sb_advance(s["ctx"], variant, 1.0, -c0, dt, steps, s["ramp"])
        return _get_state(s)
    if case["kind"] == "readout":
        return _readout(s)
    if case["kind"] == "backward":
        loss, g = sb.sb_backward(s["ctx"], 1.0, s["c0_abs"], dt, steps, R, s["seed"] + 1,
                                 s["ramp"], case["every"], s["grad"])
        return [loss, g["dt"], g["c0"], g["w_q"], g["w_c"], s["grad"]]
    q = sb.sb_qubo_build_device(s["event"], s["params"])[0]
    ctx = _context(case, [q])
    sb.sb_run(ctx, variant, 1.0, -c0, dt, steps, R, s["seed"] + 1)
    T, E, r = sb.sb_best(ctx)
    tr = sb.sb_tracks(s["event"], q, T)
    sb.sb_destroy(ctx)
    track = np.full(s["event"].n_hits, -1, np.int32)  # the track that each hit is on
    for k, t in enumerate(tr["tracks"]):
        track[t] = k
    return [T, E, r, track, tr["tp"], tr["fp"], tr["fn"], q.rowptr, q.col, q.val, q.lin]


# ---------------------------------------------------------------- what a pass cannot do without
def work(case):
    """Per SB step: the state x, y read and written (16 bytes a spin), column and
    coupling of every nonzero (once for all replicas), row pointer and field of
    every row; two operations per nonzero and replica, ten per spin. A readout
    reads x, the FP64 couplings, columns and linear terms once. A gradient step
    is a forward and a reverse step, and the reverse reads what the forward
    recorded. Event sizes are the presets' typical ones."""
    R, E = case["replicas"], case["events"]
    if E > 1:
        # mean over log-uniform track counts
        ts = [50.0 * (case["tracks"] / 50.0) ** ((i + 0.5) / 16) for i in range(16)]
        ns = [_rows(t, case["cuts"]) for t in ts]
        n = E * sum(ns) / 16
        nnz = E * sum(v * _nnz_per_row(v, case["cuts"]) for v in ns) / 16
    else:
        n = _rows(case["tracks"], case["cuts"])
        nnz = n * _nnz_per_row(n, case["cuts"])
    jb = 2 if case["prec"] == "bf16" else 4
    step_b, step_f = 16.0 * n * R + (4 + jb) * nnz + 8.0 * n, 2.0 * nnz * R + 10.0 * n * R
    read_b, read_f = 4.0 * n * R + 12.0 * nnz + 12.0 * n, 2.0 * nnz * R + 2.0 * n * R
    S = case["steps"]
    if case["kind"] == "readout":
        return {"bytes": read_b, "flops": read_f}
    if case["kind"] == "backward":
        return {"bytes": S * (2 * step_b + 17.0 * n * R), "flops": 3 * S * step_f}
    reads = -(-S // case["every"]) + 1 if case["kind"] == "trace" else 1
    if case["kind"] == "advance":
        return {"bytes": S * step_b, "flops": S * step_f}
    return {"bytes": S * step_b + reads * read_b, "flops": S * step_f + reads * read_f}


# ---------------------------------------------------------------- the same in 64 bits
def _product(q, vals):
    """Sparse matrix of the QUBO's pattern as an FP64 CSR tensor on the GPU."""
    return torch.sparse_csr_tensor(torch.from_numpy(q.rowptr.astype(np.int64)),
                                   torch.from_numpy(q.col.astype(np.int64)),
                                   torch.from_numpy(np.ascontiguousarray(vals)),
                                   size=(q.n, q.n)).cuda()


def _ising(case, q, val, lin):
    """(J as the context's precision holds it, h as FP32 holds it, sigma_J, row index)."""
    rows = np.repeat(np.arange(q.n), np.diff(q.rowptr))
    J = -val / 4.0
    h = -(lin / 2.0 + np.bincount(rows, weights=val, minlength=q.n) / 4.0)
    sigma = math.sqrt(float(np.sum(J * J)) / (q.n * (q.n - 1.0)))
    Jt = torch.from_numpy(J)
    Jt = Jt.to(torch.float32) if case["prec"] == "fp32" else Jt.to(torch.bfloat16)
    return Jt.to(torch.float64).numpy(), h.astype(np.float32).astype(np.float64), sigma


def _f32(v):
    return float(np.float32(v))


def _exact_advance(case, seed):
    qs = _qubos(case, seed)
    x, y = _state(case, seed, sum(q.n for q in qs))
    x, y = x.double(), y.double()
    ramp, dt, r0 = _ramp(case).double().tolist(), _f32(case["dt"]), 0
    dta0 = _f32(case["dt"] * 1.0)
    for q in qs:
        J, h, sigma = _ising(case, q, q.val, q.lin)
        c0 = _f32(case["c0"] * 0.5 / (math.sqrt(q.n) * sigma))
        J, h = _product(q, J), torch.from_numpy(h).cuda()[:, None]
        xe, ye = x[r0:r0 + q.n], y[r0:r0 + q.n]
        for a in ramp:
            f = J @ (torch.sign(xe) if case["variant"] == "dsb" else xe)
            force = -(1.0 - a) * xe + c0 * (f + h)
            if case["variant"] == "asb":
                force -= xe * xe * xe
            ye = ye + dt * force
            xe = xe + dta0 * ye
            if case["variant"] != "asb":
                wall = xe.abs() > 1.0
                xe = torch.where(wall, torch.sign(xe), xe)
                ye = torch.where(wall, 0.0, ye)
        x[r0:r0 + q.n], y[r0:r0 + q.n] = xe, ye
        r0 += q.n
    return [x, y]


def _exact_readout(case, seed):
    qs = _qubos(case, seed)
    x, _ = _state(case, seed, sum(q.n for q in qs))
    Es, r0 = [], 0
    for q in qs:
        T = (x[r0:r0 + q.n] > 0).double()
        lin = torch.from_numpy(q.lin).cuda()
        Es.append(lin @ T + 0.5 * (T * (_product(q, q.val) @ T)).sum(0))
        r0 += q.n
    E = torch.stack(Es)
    return [E, E.min(1).values, None, None]


_PHILOX_M = (0xD2511F53, 0xCD9E8D57)
_PHILOX_W = (0x9E3779B9, 0xBB67AE85)


def _philox_start(seed, n, R):
    """x, y of the start: Philox4x32-10 (Salmon et al. 2011), counter (row,
    replica, 3, 0), key = seed; the top 24 bits of words 0 and 1 to U(-0.01, 0.01)."""
    u64, m32 = np.uint64, np.uint64(0xFFFFFFFF)
    c = [np.repeat(np.arange(n, dtype=u64), R), np.tile(np.arange(R, dtype=u64), n),
         np.full(n * R, 3, u64), np.zeros(n * R, u64)]
    k = [seed & 0xFFFFFFFF, (seed >> 32) & 0xFFFFFFFF]
    for _ in range(10):
        p0, p1 = c[0] * u64(_PHILOX_M[0]), c[2] * u64(_PHILOX_M[1])
        c = [(p1 >> u64(32)) ^ c[1] ^ u64(k[0]), p1 & m32, (p0 >> u64(32)) ^ c[3] ^ u64(k[1]),
             p0 & m32]
        k = [(k[0] + _PHILOX_W[0]) & 0xFFFFFFFF, (k[1] + _PHILOX_W[1]) & 0xFFFFFFFF]
    return c[0], c[1]


def _exact_backward(case, seed):
    q = _qubos(case, seed)[0]
    R, S, n = case["replicas"], case["steps"], q.n
    val, lin = np.where(q.cls == 0, -1.0, 1.0), 1.0 * q.quality
    Jv, hv, sigma = _ising(case, q, val, lin)
    c0 = _f32(case["c0"] * 0.5 / (math.sqrt(n) * sigma))
    dt, ramp = _f32(case["dt"]), _ramp(case).double().tolist()
    J, C = _product(q, Jv), _product(q, (q.cls == 1).astype(np.float64))
    h = torch.from_numpy(hv).cuda()[:, None]
    quality = torch.from_numpy(q.quality).cuda()
    nconf = torch.from_numpy(np.bincount(np.repeat(np.arange(n), np.diff(q.rowptr)),
                                         weights=(q.cls == 1).astype(np.float64),
                                         minlength=n)).cuda()
    x, y = (torch.from_numpy(_start_value(w).reshape(n, R)).cuda()
            for w in _philox_start(seed + 1, n, R))
    xs, yts, keeps, fs = [x], [], [], []
    for a in ramp:
        f = J @ x
        yt = y + dt * (-(1.0 - a) * x + c0 * (f + h))
        xt = x + dt * yt
        keep = xt.abs() <= 1.0
        x, y = torch.where(keep, xt, torch.sign(xt)), torch.where(keep, yt, 0.0)
        xs.append(x)
        yts.append(yt)
        keeps.append(keep)
        fs.append(f)
    Jx = J @ x
    loss = float((-0.5 * x * Jx - h * x).sum()) / R
    lx, ly = (-Jx - h) / R, torch.zeros_like(x)
    gh = -x.sum(1) / R
    g_wc = float((x * (C @ x)).sum()) / (8.0 * R)
    g_dt = g_c0 = 0.0
    g_a = torch.zeros(S, dtype=torch.float64, device="cuda")
    for k in range(S - 1, -1, -1):
        lxt = torch.where(keeps[k], lx, 0.0)
        lyt = torch.where(keeps[k], ly, 0.0) + dt * lxt
        xk, f = xs[k], fs[k]
        g_dt += float((lyt * (-(1.0 - ramp[k]) * xk + c0 * (f + h))).sum()
                      + (lxt * yts[k]).sum())
        g_c0 += float((lyt * dt * (f + h)).sum())
        g_a[k] = (lyt * dt * xk).sum()
        gh += dt * c0 * lyt.sum(1)
        g_wc += float((dt * c0 * lyt * (-0.25) * (C @ xk)).sum())
        lx = lxt - dt * (1.0 - ramp[k]) * lyt + dt * c0 * (J @ lyt)
        ly = lyt
    return [loss, g_dt, g_c0, float((gh * (-quality / 2.0)).sum()),
            g_wc + float((gh * (-nconf / 4.0)).sum()), g_a]


def _start_value(w):
    """U(-0.01, 0.01) of a Philox word, as the FP32 start has it."""
    v = (w >> np.uint64(8)).astype(np.int64) - (1 << 23)
    return (v.astype(np.float32) * np.float32(0.01 / (1 << 23))).astype(np.float64)


def exact(case, seed):
    """"run", "trace" and "solve" have no such value: over hundreds of steps the
    trajectories of a bifurcating system part from any other rounding, and a
    solve's outputs are selections, whole numbers and the builder's values."""
    if case["kind"] == "advance":
        return _exact_advance(case, seed)
    if case["kind"] == "readout":
        return _exact_readout(case, seed)
    if case["kind"] == "backward":
        return _exact_backward(case, seed)
    return None
