"""Performance cases: the work a user of this framework has it do, through its public entry points.

``listed()`` gives the standing cases, ``draw(rng)`` further ones of the same ranges.  ``prepare`` makes what a
program holds before the call (inputs, weights, a context with a filled replay buffer), ``run`` is one pass,
``work`` the bytes and operations the pass cannot do without, and ``exact`` the same outputs in 64 bits, written
here from the method's definition in plain torch / numpy.

Kinds of case and what they stand for:

* ``relabel``: one call of the hindsight sampler (``CRLContext.sample``) on a full replay buffer.
* ``loss``: the critic objective behind autograd (``functional.infonce_loss``), forward and backward.
* ``encoder``: one network behind autograd (``functional.encoder``), forward and backward with the gradients of
  its parameters and of its second input (the action the policy is trained through).
* ``critic``: one critic step with its Adam update on a given batch (``CRLContext.critic_step``).
* ``collect``: an unroll of environment steps with the policy (``CRLContext.collect``).
* ``update``: a whole update step (insert one time slice, relabel, critic, actor, Adam) on a side stream, where the
  library replays it as a graph.
* ``sweep``: the same step for many independent agents of uneven shapes in grouped launches (``CRLSweep``).
"""

import math

import numpy as np
import torch

from paper_2408_11052_gb300 import api, functional, workload

ANT = dict(D=29, A=8, G=2)
HUMANOID = dict(D=268, A=17, G=3)
STRESS = dict(D=64, A=16, G=8)


def listed():
    return [
        # the smallest call: one Ant batch drawn from a full buffer of 1024 environments
        dict(name="relabel_ant", kind="relabel", E=1024, T=1000, B=256, **ANT),
        # sampling throughput on Humanoid rows (an epoch's worth of transitions in one call)
        dict(name="relabel_humanoid_1m", kind="relabel", E=1024, T=1000, B=1 << 20, **HUMANOID),
        # the critic objective at the paper's default batch, where latency and launches count
        dict(name="loss_ant_bf16", kind="loss", precision="bf16", B=256, R=64, energy="l2", loss="sym"),
        # the large-batch contrastive objective
        dict(name="loss_large_bf16", kind="loss", precision="bf16", B=8192, R=256, energy="l2", loss="fwd"),
        # the objective with the wrapper's default (plain FP32) path at a batch that fits no tile
        dict(name="loss_ragged_fp32", kind="loss", precision="fp32", B=1001, R=64, energy="l2", loss="sym"),
        # the deep LayerNorm encoder of the Humanoid runs
        dict(name="encoder_humanoid_bf16", kind="encoder", precision="bf16", B=1024, in0=268, in1=17, hidden=1024,
             layers=4, out=64, layernorm=True),
        # the encoder of the large-batch runs
        dict(name="encoder_large_bf16", kind="encoder", precision="bf16", B=8192, in0=64, in1=16, hidden=512, layers=2,
             out=256, layernorm=False),
        # the small FP32 critic step (a context's default precision)
        dict(name="critic_small_fp32", kind="critic", precision="fp32", B=256, hidden=256, layers=2, R=64,
             layernorm=False, energy="l2", loss="sym", **ANT),
        # one unroll of the collection loop: 62 steps of 1024 environments
        dict(name="collect_ant", kind="collect", E=1024, n=62, hidden=256, layers=2, layernorm=False, **ANT),
        # the whole step at the paper's default sizes
        dict(name="update_ant_bf16", kind="update", E=1024, T=1000, B=256, hidden=256, layers=2, R=64,
             layernorm=False, energy="l2", loss="sym", **ANT),
        # the whole step at the large batch
        dict(name="update_large_bf16", kind="update", E=4096, T=500, B=8192, hidden=512, layers=2, R=256,
             layernorm=False, energy="l2", loss="fwd", **STRESS),
        # 32 agents with uneven batches and observation sizes advanced together
        dict(name="sweep_32_bf16", kind="sweep", agents=32, E=512, T=200),
    ]


def _log_int(rng, lo, hi, step=1):
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return max(lo, min(hi, int(round(v / step)) * step))


def draw(rng):
    kind = rng.choice(["relabel", "loss", "loss", "encoder", "encoder", "critic", "collect", "update", "update", "sweep"])
    env = dict(rng.choice([ANT, HUMANOID, STRESS, dict(D=rng.randint(8, 120), A=rng.randint(3, 20), G=rng.randint(2, 8))]))
    if kind == "relabel":
        E, T = _log_int(rng, 64, 2048), _log_int(rng, 100, 1000)
        top = (1 << 20) * 288 // max(288, env["D"] + env["A"])
        return dict(kind=kind, E=E, T=T, B=_log_int(rng, 256, top), **env)
    if kind == "loss":
        precision = rng.choice(["bf16", "bf16", "fp32"])
        loss = rng.choice(["sym", "sym", "fwd", "bwd", "flatnce_fwd", "nce_binary", "dpo"])
        energy = rng.choice(["l2", "l2", "cos", "dot", "l2sq", "l1"])
        if precision == "fp32":
            return dict(kind=kind, precision=precision, B=_log_int(rng, 64, 2048), R=_log_int(rng, 16, 256),
                        energy=energy, loss=loss)
        top = 1024 if energy == "l1" else 8192 if loss in ("sym", "fwd", "bwd", "flatnce_fwd") else 4096
        return dict(kind=kind, precision=precision, B=_log_int(rng, 64, top, 8), R=rng.choice([64, 128, 192, 256]),
                    energy=energy, loss=loss)
    if kind == "encoder":
        precision = rng.choice(["bf16", "bf16", "fp32"])
        hidden = _log_int(rng, 64, 1024 if precision == "bf16" else 512, 8)
        layers = rng.randint(1, 4)
        top = 8192 if hidden <= 512 and layers <= 2 else 2048
        return dict(kind=kind, precision=precision, B=_log_int(rng, 64, top if precision == "bf16" else 1024),
                    in0=env["D"], in1=env["A"], hidden=hidden, layers=layers, out=rng.choice([64, 128, 256]),
                    layernorm=rng.random() < 0.4)
    if kind == "critic":
        precision = rng.choice(["fp32", "bf16"])
        return dict(kind=kind, precision=precision, B=_log_int(rng, 64, 1024, 1 if precision == "fp32" else 8),
                    hidden=_log_int(rng, 64, 512, 8), layers=rng.randint(2, 3), R=rng.choice([64, 128]),
                    layernorm=rng.random() < 0.3, energy=rng.choice(["l2", "cos", "dot"]),
                    loss=rng.choice(["sym", "fwd", "bwd"]), **env)
    if kind == "collect":
        return dict(kind=kind, E=_log_int(rng, 64, 1024), n=_log_int(rng, 8, 62), hidden=_log_int(rng, 64, 256, 8),
                    layers=2, layernorm=rng.random() < 0.3, **env)
    if kind == "update":
        B = _log_int(rng, 64, 4096, 8)
        deep = B <= 1024 and rng.random() < 0.4
        return dict(kind=kind, E=_log_int(rng, 128, 1024), T=_log_int(rng, 100, 500), B=B,
                    hidden=1024 if deep else _log_int(rng, 128, 512, 8), layers=4 if deep else 2,
                    R=rng.choice([64, 128, 256]), layernorm=deep, energy=rng.choice(["l2", "cos", "dot"]),
                    loss=rng.choice(["sym", "fwd", "bwd"]), **env)
    return dict(kind=kind, agents=_log_int(rng, 2, 32), E=_log_int(rng, 64, 512), T=_log_int(rng, 50, 200))


# ---- shapes -----------------------------------------------------------------------------------------------------
def _dims(n_in, hidden, layers, out):
    return [n_in] + [hidden] * layers + [out]


def _layout(dims, layernorm):
    """The documented flat layout: per layer W [out][in], b, then gain and shift; each tensor at a multiple of 64."""
    off, lay = 0, []
    for i in range(len(dims) - 1):
        sizes = [dims[i + 1] * dims[i], dims[i + 1]]
        if layernorm and i < len(dims) - 2:
            sizes += [dims[i + 1], dims[i + 1]]
        at = []
        for n in sizes:
            at.append((off, n))
            off += (n + 63) // 64 * 64
        lay.append(at)
    return off, lay


def _work_of(case):
    """A workload of the library for the cases that run on a context."""
    c = case
    return workload.Workload(c["kind"], E=c.get("E", 64), T=c.get("T", 8), D=c["D"], A=c["A"], G=c["G"], B=c.get("B", 64),
                             hidden=c.get("hidden", 64), layers=c.get("layers", 2), repr=c.get("R", 64),
                             layernorm=c.get("layernorm", False), energy=c.get("energy", "l2"),
                             loss=c.get("loss", "sym"), episode_len=min(1000, c.get("T", 1000)))


def _nets(w):
    return {"phi": _dims(w.D + w.A, w.hidden, w.layers, w.repr), "psi": _dims(w.G, w.hidden, w.layers, w.repr),
            "pi": _dims(w.D + w.G, w.hidden, w.layers, 2 * w.A)}


# ---- inputs -----------------------------------------------------------------------------------------------------
def _gen(seed, salt):
    g = torch.Generator(device="cuda")
    g.manual_seed(1_000_003 * int(seed) + salt)
    return g


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device="cuda")


def _params(g, dims, layernorm):
    """Flat parameters: W ~ N(0, 1 / fan_in), small biases, gains near 1 (a network some way into its training)."""
    n, lay = _layout(dims, layernorm)
    p = torch.zeros(n, device="cuda")
    for i, at in enumerate(lay):
        for k, (o, m) in enumerate(at):
            p[o:o + m] = _randn(g, m) * (1.0 / math.sqrt(dims[i]) if k == 0 else 0.1)
            if k == 2:
                p[o:o + m] += 1.0
    return p


def _trajectories(g, w, n):
    """n time slices of every environment: random-walk states with fixed-length episodes, uniform actions."""
    t = torch.arange(n, device="cuda")
    done = ((t + 1) % w.episode_len == 0).to(torch.uint8)[:, None].expand(n, w.E).contiguous()
    act = torch.rand(n, w.E, w.A, generator=g, device="cuda") * 2 - 1
    obs = _randn(g, n, w.E, w.D)
    for t0 in range(0, n, w.episode_len):
        obs[t0 + 1:t0 + w.episode_len] *= 0.1
        obs[t0:t0 + w.episode_len] = torch.cumsum(obs[t0:t0 + w.episode_len], dim=0)
    return obs, act, done


def _batch(g, w):
    """A relabelled batch: states and actions, and goals a few random-walk steps away from their states."""
    s = _randn(g, w.B, w.D)
    a = torch.rand(w.B, w.A, generator=g, device="cuda") * 2 - 1
    return s, a, (s[:, :w.G] + 0.5 * _randn(g, w.B, w.G)).contiguous()


def _representations(g, case):
    """phi, psi [B][R]: positive pairs closer than the others; rows scaled so that every energy stays O(10)."""
    B, R = case["B"], case["R"]
    phi = _randn(g, B, R)
    psi = 0.6 * phi + 0.8 * _randn(g, B, R)
    k = {"dot": R ** -0.25, "l2sq": R ** -0.5, "l1": 8.0 / R}.get(case["energy"], 1.0)
    return phi * k, psi * k


_SLICES = 4    # further time slices an update case inserts, one per pass (in turn)
_POLICIES = 30    # a sweep's pass returns every agent's phi and this many policies (64 outputs at most)


def _sweep_workloads(case, seed):
    ws = workload.sweep_agents(case["agents"], seed=4)
    return [w.with_(E=case["E"], T=case["T"], episode_len=case["T"], seed=(seed * 64 + i) % (1 << 31))
            for i, w in enumerate(ws)]


def _fill(ctx, w, g):
    """A context's weights and a full replay buffer."""
    for net, dims in _nets(w).items():
        ctx.store[net]["params"].copy_(_params(g, dims, w.layernorm))
    obs, act, done = _trajectories(g, w, w.T)
    ctx.insert(obs, act, done)
    return obs, act, done


def _slices(g, w):
    return (_randn(g, _SLICES, w.E, w.D), torch.rand(_SLICES, w.E, w.A, generator=g, device="cuda") * 2 - 1,
            torch.zeros(_SLICES, w.E, dtype=torch.uint8, device="cuda"))


_side = []


def _stream():
    """The program's training stream: one for all states, as steps follow one another (not the default stream, which
    cannot be captured)."""
    if not _side:
        _side.append(torch.cuda.Stream())
    return _side[0]


def prepare(case, seed):
    kind = case["kind"]
    g = _gen(seed, 1)
    if kind == "loss":
        phi, psi = _representations(g, case)
        return dict(case=case, phi=phi.requires_grad_(True), psi=psi.requires_grad_(True))
    if kind == "encoder":
        c = case
        p = _params(g, _dims(c["in0"] + c["in1"], c["hidden"], c["layers"], c["out"]), c["layernorm"])
        x0, x1 = _randn(g, c["B"], c["in0"]), torch.rand(c["B"], c["in1"], generator=g, device="cuda") * 2 - 1
        return dict(case=case, p=p.requires_grad_(True), x0=x0, x1=x1.requires_grad_(True),
                    dy=_randn(g, c["B"], c["out"]) / c["B"])
    if kind == "sweep":
        ws = _sweep_workloads(case, seed)
        stream = _stream()
        with torch.cuda.stream(stream):
            sweep = api.CRLSweep(ws)
            more = []
            for i, (w, ctx) in enumerate(zip(ws, sweep.agents)):
                _fill(ctx, w, _gen(seed, 10 + i))
                more.append(_slices(_gen(seed, 100 + i), w))
        stream.synchronize()
        return dict(case=case, sweep=sweep, stream=stream, more=more, at=0,
                    loss=torch.zeros(len(ws), 6, device="cuda"))
    w = _work_of(case).with_(seed=int(seed) % (1 << 31))
    if kind == "update":
        stream = _stream()
        with torch.cuda.stream(stream):
            ctx = api.CRLContext(w, precision="bf16", path="fused")
            _fill(ctx, w, g)
            more = _slices(_gen(seed, 2), w)
        stream.synchronize()
        return dict(case=case, ctx=ctx, stream=stream, more=more, at=0, loss=torch.zeros(6, device="cuda"))
    if kind == "critic":
        ctx = api.CRLContext(w, precision=case["precision"], path="fused" if case["precision"] == "bf16" else "plain")
        for net, dims in _nets(w).items():
            ctx.store[net]["params"].copy_(_params(g, dims, w.layernorm))
        return dict(case=case, ctx=ctx, batch=_batch(g, w), loss=torch.zeros(4, device="cuda"))
    if kind == "collect":
        w = w.with_(T=max(case["n"], 64))
        ctx = api.CRLContext(w, precision="bf16", path="fused")
        ctx.store["pi"]["params"].copy_(_params(g, _nets(w)["pi"], w.layernorm))
        n, E = case["n"], case["E"]
        return dict(case=case, ctx=ctx, out=(torch.zeros(n, E, w.D, device="cuda"), torch.zeros(n, E, w.A, device="cuda"),
                                             torch.zeros(n, E, dtype=torch.uint8, device="cuda")))
    ctx = api.CRLContext(w.with_(B=64))    # the sampler takes any batch size
    obs, act, done = _trajectories(g, w, w.T)
    ctx.insert(obs, act, done)
    return dict(case=case, ctx=ctx, step=0)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "relabel":
        step = state["step"]
        state["step"] += 1
        return dict(zip(("s", "a", "g", "idx"), state["ctx"].sample(step, B=case["B"])))
    if kind == "loss":
        total, parts = functional.infonce_loss(state["phi"], state["psi"], energy=case["energy"], loss=case["loss"],
                                               path="fused" if case["precision"] == "bf16" else "plain")
        dphi, dpsi = torch.autograd.grad(total, (state["phi"], state["psi"]))
        return dict(parts=parts, dphi=dphi, dpsi=dpsi)
    if kind == "encoder":
        y = functional.encoder(state["p"], state["x0"], state["x1"], case["in0"], case["in1"], case["hidden"],
                               case["layers"], case["out"], case["layernorm"],
                               precision="bf16" if case["precision"] == "bf16" else None)
        dp, dx1 = torch.autograd.grad(y, (state["p"], state["x1"]), state["dy"])
        return dict(y=y, dparams=dp, dx1=dx1)
    if kind == "critic":
        ctx = state["ctx"]
        s, a, g = state["batch"]
        ctx.critic_step(s, a, g, apply_update=True, loss_out=state["loss"])
        return dict(loss=state["loss"], **{net + "_" + k: ctx.store[net][k] for net in ("phi", "psi")
                                           for k in ("params", "grads")})
    if kind == "collect":
        state["ctx"].collect(case["n"], episode_length=1000, out=state["out"])
        return dict(zip(("obs", "act", "done"), state["out"]))
    i = state["at"]
    state["at"] = (i + 1) % _SLICES
    with torch.cuda.stream(state["stream"]):
        if kind == "update":
            ctx = state["ctx"]
            ctx.update_step(*(x[i:i + 1] for x in state["more"]), loss_out=state["loss"])
            return dict(loss=state["loss"], **{net + "_" + k: ctx.store[net][k] for net in api.NET
                                               for k in ("params", "grads")})
        sweep = state["sweep"]
        sweep.update_step(*([m[k][i:i + 1] for m in state["more"]] for k in range(3)), loss_out=state["loss"])
        return dict(loss=state["loss"], phi=[a.store["phi"]["params"] for a in sweep.agents],
                    pi=[a.store["pi"]["params"] for a in sweep.agents[:_POLICIES]])


# ---- work -------------------------------------------------------------------------------------------------------
def _mlp_work(M, dims, backward, dx=False):
    """Operations of one network's passes, and the bytes of its parameters."""
    pairs = sum(dims[i] * dims[i + 1] for i in range(len(dims) - 1))
    flops = 2.0 * M * pairs
    if backward:
        flops += 2.0 * M * pairs + 2.0 * M * (pairs - (0 if dx else dims[0] * dims[1]))
    return flops, 4.0 * pairs


def _update_work(w):
    """The critic and actor passes of one step with Adam: forward and backward of phi and psi, the energy matrix and
    its two gradient products, then pi, phi and psi forward, the input gradient of phi and the backward of pi."""
    n = _nets(w)
    flops, bytes_ = 6.0 * w.B * w.B * w.repr, 0.0
    for net in ("phi", "psi", "pi"):
        f, b = _mlp_work(w.B, n[net], True)
        flops += f
        bytes_ += 6 * b                                 # parameters and moments read and written
    flops += _mlp_work(w.B, n["phi"], False)[0] * 2 + _mlp_work(w.B, n["psi"], False)[0]
    return flops, bytes_ + 4.0 * w.B * (w.D + w.A + w.G) + 8.0 * w.E * (w.D + w.A)


def work(case):
    kind = case["kind"]
    if kind == "relabel":
        D, A, G, B = (case[k] for k in "DAGB")
        return {"bytes": B * (4.0 * (D + A + 1 + G) + 4.0 * (D + A + G + 3)), "flops": 0.0}
    if kind == "loss":
        B, R = case["B"], case["R"]
        return {"bytes": 16.0 * B * R, "flops": 6.0 * B * B * R}
    if kind == "encoder":
        dims = _dims(case["in0"] + case["in1"], case["hidden"], case["layers"], case["out"])
        f, b = _mlp_work(case["B"], dims, True, dx=True)
        return {"bytes": 2 * b + 4.0 * case["B"] * (dims[0] + 2 * dims[-1] + case["in1"]), "flops": f}
    if kind == "sweep":
        both = [_update_work(w) for w in _sweep_workloads(case, 0)]
        return {"bytes": sum(b for _, b in both), "flops": sum(f for f, _ in both)}
    w = _work_of(case)
    if kind == "critic":
        (fp, bp), (fq, bq) = (_mlp_work(w.B, _nets(w)[n], True) for n in ("phi", "psi"))
        return {"bytes": 7 * (bp + bq) + 4.0 * w.B * (w.D + w.A + w.G), "flops": fp + fq + 6.0 * w.B * w.B * w.repr}
    if kind == "collect":
        f, b = _mlp_work(case["E"], _nets(w)["pi"], False)
        return {"bytes": b + case["n"] * case["E"] * 8.0 * (w.D + w.A), "flops": case["n"] * f}
    f, b = _update_work(w)
    return {"bytes": b, "flops": f}


# ---- the same in 64 bits ----------------------------------------------------------------------------------------
_U = np.uint64
_LOW = _U(0xFFFFFFFF)


def _mul_hi_lo(a, b):
    """High and low words of the 128-bit products of uint64 values."""
    a, b = np.asarray(a, dtype=_U), np.asarray(b, dtype=_U)
    s = _U(32)
    a0, a1, b0, b1 = a & _LOW, a >> s, b & _LOW, b >> s
    p00, p01, p10, p11 = a0 * b0, a0 * b1, a1 * b0, a1 * b1
    mid = (p00 >> s) + (p01 & _LOW) + (p10 & _LOW)
    return p11 + (p01 >> s) + (p10 >> s) + (mid >> s), a * b


def _philox(c0, c1, c2, c3, seed, agent):
    """Philox4x64-10 (Salmon et al., SC'11) for arrays of counters."""
    with np.errstate(over="ignore"):
        x = [v.copy() for v in np.broadcast_arrays(*(np.asarray(c, dtype=_U) for c in (c0, c1, c2, c3)))]
        k0, k1 = _U(seed), _U(agent)
        for _ in range(10):
            h0, l0 = _mul_hi_lo(x[0], _U(0xD2E7470EE14C6C93))
            h1, l1 = _mul_hi_lo(x[2], _U(0xCA5A826395121157))
            x = [h1 ^ x[1] ^ k0, l1, h0 ^ x[3] ^ k1, l0]
            k0, k1 = k0 + _U(0x9E3779B97F4A7C15), k1 + _U(0xBB67AE8584CAA73B)
    return x


def _normals(seed, agent, step, B, n, word):
    """[B][n] standard normals: Box-Muller on the words of block (step, b, word, d / 4)."""
    b, q = np.meshgrid(np.arange(B), np.arange((n + 3) // 4), indexing="ij")
    w = _philox(step, b, word, q, seed, agent)
    u = [((v >> _U(11)).astype(np.float64) + 0.5) * 2.0 ** -53 for v in w]
    cols = []
    for p in (0, 2):
        rad, ang = np.sqrt(-2.0 * np.log(u[p])), 2.0 * np.pi * u[p + 1]
        cols += [rad * np.cos(ang), rad * np.sin(ang)]
    return torch.from_numpy(np.stack(cols, axis=-1).reshape(B, -1)[:, :n].copy()).cuda()


def _draw_batch(w, agent, obs, act, done, step, B):
    """The relabelled batch of a step: (s, a, g) in 64 bits and idx [B][3] = (environment, time, offset)."""
    size = obs.shape[0]
    word = _philox(step, np.arange(B), 0, 0, w.seed, agent)
    idx = _mul_hi_lo(word[0], _U(w.E * size))[0].astype(np.int64)
    e, t = idx // size, idx % size
    # the last step of the episode of (t, e), at most the newest stored one
    d = done.cpu().numpy().astype(bool)
    end = np.full((size, w.E), size - 1, dtype=np.int64)
    for i in range(size - 2, -1, -1):
        end[i] = end[i + 1]
        end[i][d[i]] = i
    end[size - 1] = size - 1
    left = end[t, e] - t
    # gamma^k in 32-bit fixed point; C[j] = 2^32 (1 - gamma^j)
    gq = int(math.floor(float(np.float32(w.gamma)) * 2.0 ** 32 + 0.5))
    table = [1 << 32]
    for _ in range(w.T + 1):
        table.append((table[-1] * gq) >> 32)
    C = np.array([(1 << 32) - x for x in table], dtype=_U)
    q = ((word[1] >> _U(32)) * C[left]) >> _U(32)
    k = np.where(left > 0, np.searchsorted(C, q, side="right"), 0)
    te, ee, ke = (torch.from_numpy(x).cuda() for x in (t, e, k))
    return (obs[te, ee].double(), act[te, ee].double(), obs[te + ke, ee][:, :w.G].double(),
            torch.stack([ee, te, ke], dim=1).int())


def _forward(p, x, dims, layernorm):
    _, lay = _layout(dims, layernorm)
    for i, at in enumerate(lay):
        t = [p[o:o + n] for o, n in at]
        x = x @ t[0].view(dims[i + 1], dims[i]).T + t[1]
        if i < len(lay) - 1:
            if layernorm:
                x = torch.nn.functional.layer_norm(x, (dims[i + 1],), t[2], t[3], eps=1e-6)
            x = torch.relu(x)
    return x


def _energies(phi, psi, energy):
    """F [B][B] in blocks of rows (the distances from differences, not from the expanded square)."""
    if energy == "dot":
        return phi @ psi.T
    if energy == "cos":
        return (phi / phi.norm(dim=1, keepdim=True)) @ (psi / psi.norm(dim=1, keepdim=True)).T
    if energy == "l1":
        return -torch.cdist(phi, psi, p=1.0)
    d2 = (phi * phi).sum(1)[:, None] + (psi * psi).sum(1)[None] - 2.0 * phi @ psi.T
    d2 = d2.clamp_min(0.0)
    return -d2 if energy == "l2sq" else -torch.sqrt(d2)


_BETA = float(np.float32(0.1))


def _objective(phi, psi, energy, loss):
    """The value whose gradient is taken, and the reported parts (total, forward, backward, penalty)."""
    F = _energies(phi, psi, energy)
    B = F.shape[0]
    r, c, d = torch.logsumexp(F, 1), torch.logsumexp(F, 0), torch.diagonal(F)
    fwd, bwd = (r - d).mean(), (c - d).mean()
    penalty = _BETA * (r * r).mean()
    sp = torch.nn.functional.softplus
    if loss == "fwd":
        value = shown = fwd
    elif loss == "bwd":
        value = shown = bwd
    elif loss == "sym":
        value = shown = 0.5 * (fwd + bwd)
    elif loss == "flatnce_fwd":
        value, shown = fwd, torch.zeros_like(fwd)      # value 0, the gradient of mean_i log S_i
    elif loss == "dpo":
        value = shown = sp(F - d[:, None]).mean()
    else:                                              # nce_binary
        value = shown = (sp(F).sum() - d.sum()) / (B * B)
    return value + penalty, torch.stack([shown + penalty, fwd, bwd, penalty]).detach()


def _adam(p, g, lr):
    """The first Adam step from zero moments."""
    b1, b2, eps = (float(np.float32(x)) for x in (0.9, 0.999, 1e-8))
    m, v = (1 - b1) * g, (1 - b2) * g * g
    return p - lr * (m / (1 - b1)) / (torch.sqrt(v / (1 - b2)) + eps)


def _critic64(w, p, s, a, g):
    """(loss parts, gradients, updated parameters) of the critic step on flat 64-bit parameters."""
    n = _nets(w)
    pp, pq = (p[k].clone().requires_grad_(True) for k in ("phi", "psi"))
    phi = _forward(pp, torch.cat([s, a], 1), n["phi"], w.layernorm)
    psi = _forward(pq, g, n["psi"], w.layernorm)
    total, parts = _objective(phi, psi, w.energy, w.loss)
    gp, gq = torch.autograd.grad(total, (pp, pq))
    lr = float(np.float32(w.lr_critic))
    return parts, {"phi": gp, "psi": gq}, {"phi": _adam(p["phi"], gp, lr), "psi": _adam(p["psi"], gq, lr)}


def _policy(out, eps):
    A = out.shape[1] // 2
    ell = out[:, A:].clamp(-5.0, 2.0)
    u = out[:, :A] + torch.exp(ell) * eps
    logpi = (-0.5 * eps * eps - 0.5 * math.log(2 * math.pi) - ell
             - 2.0 * (math.log(2.0) - u - torch.nn.functional.softplus(-2.0 * u))).sum(1)
    return torch.tanh(u), logpi


def _update64(w, agent, params, obs, act, done):
    """Losses, gradients and parameters after the first update step of a fresh context."""
    p = {k: v.double() for k, v in params.items()}
    s, a, g, _ = _draw_batch(w, agent, obs, act, done, 0, w.B)
    parts, grads, new = _critic64(w, p, s, a, g)
    n = _nets(w)
    pi = p["pi"].clone().requires_grad_(True)
    eps = _normals(w.seed, agent, 0, w.B, w.A, 1)
    a_new, logpi = _policy(_forward(pi, torch.cat([s, g], 1), n["pi"], w.layernorm), eps)
    phi = _forward(new["phi"], torch.cat([s, a_new], 1), n["phi"], w.layernorm)
    psi = _forward(new["psi"], g, n["psi"], w.layernorm)
    f = {"l2": lambda: -(phi - psi).norm(dim=1), "dot": lambda: (phi * psi).sum(1),
         "cos": lambda: torch.nn.functional.cosine_similarity(phi, psi, dim=1, eps=0.0)}[w.energy]()
    loss = (float(np.float32(w.alpha)) * logpi - f).mean()
    grads["pi"], = torch.autograd.grad(loss, pi)
    new["pi"] = _adam(p["pi"], grads["pi"], float(np.float32(w.lr_actor)))
    return torch.cat([parts, torch.stack([loss, logpi.mean()]).detach()]), grads, new


def _after_insert(g, g_more, w):
    """A context's parameters and its buffer after the first pass's insert, from the generators of prepare()."""
    params = {net: _params(g, dims, w.layernorm) for net, dims in _nets(w).items()}
    now, more = _trajectories(g, w, w.T), _slices(g_more, w)
    return params, [torch.cat([x, m[:1]])[1:] for x, m in zip(now, more)]


def exact(case, seed):
    kind = case["kind"]
    g = _gen(seed, 1)
    if kind == "loss":
        phi, psi = (x.double().requires_grad_(True) for x in _representations(g, case))
        if case["energy"] == "l1" and case["B"] > 2048:
            return None
        total, parts = _objective(phi, psi, case["energy"], case["loss"])
        dphi, dpsi = torch.autograd.grad(total, (phi, psi))
        return dict(parts=parts, dphi=dphi, dpsi=dpsi)
    if kind == "encoder":
        st = prepare(case, seed)
        p, x0, x1 = st["p"].detach().double().requires_grad_(True), st["x0"].double(), st["x1"].detach().double()
        x1.requires_grad_(True)
        dims = _dims(case["in0"] + case["in1"], case["hidden"], case["layers"], case["out"])
        y = _forward(p, torch.cat([x0, x1], 1), dims, case["layernorm"])
        dp, dx1 = torch.autograd.grad(y, (p, x1), st["dy"].double())
        return dict(y=y.detach(), dparams=dp, dx1=dx1)
    if kind == "sweep":
        steps = []
        for i, w in enumerate(_sweep_workloads(case, seed)):
            params, now = _after_insert(_gen(seed, 10 + i), _gen(seed, 100 + i), w)
            steps.append(_update64(w, i, params, *now))
        return dict(loss=torch.stack([loss for loss, _, _ in steps]), phi=[new["phi"] for _, _, new in steps],
                    pi=[new["pi"] for _, _, new in steps[:_POLICIES]])
    w = _work_of(case).with_(seed=int(seed) % (1 << 31))
    if kind == "update":
        params, now = _after_insert(g, _gen(seed, 2), w)
        loss, grads, new = _update64(w, 0, params, *now)
        return dict(loss=loss, **{net + "_" + k: v[net] for net in ("phi", "psi", "pi")
                                  for k, v in (("params", new), ("grads", grads))})
    if kind == "critic":
        p = {net: _params(g, dims, w.layernorm).double() for net, dims in _nets(w).items()}
        parts, grads, new = _critic64(w, p, *(x.double() for x in _batch(g, w)))
        return dict(loss=parts, **{net + "_" + k: v[net] for net in ("phi", "psi")
                                   for k, v in (("params", new), ("grads", grads))})
    if kind == "collect":
        return _collect64(case, w, _params(g, _nets(w)["pi"], w.layernorm).double())
    obs, act, done = _trajectories(g, w, w.T)
    return dict(zip(("s", "a", "g", "idx"), _draw_batch(w, 0, obs, act, done, 0, case["B"])))


def _collect64(case, w, pi):
    """The collection loop from its definition: policy, slice, synthetic dynamics (no episode ends within it)."""
    E, n, dims = case["E"], case["n"], _nets(w)["pi"]
    init = (1 << 64) - 1
    s, g = _normals(w.seed, 0, init, E, w.D, 4), _normals(w.seed, 0, init, E, w.G, 5)
    cols = torch.arange(w.D, device="cuda") % w.A
    obs, act = [], []
    for k in range(n):
        a, _ = _policy(_forward(pi, torch.cat([s, g], 1), dims, w.layernorm), _normals(w.seed, 0, k, E, w.A, 2))
        obs.append(s)
        act.append(a)
        s = s + 0.1 * _normals(w.seed, 0, k, E, w.D, 3) + 0.05 * a[:, cols]
    return dict(obs=torch.stack(obs), act=torch.stack(act), done=torch.zeros(n, E, dtype=torch.uint8, device="cuda"))
