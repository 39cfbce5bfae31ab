"""The workloads that this framework is timed on, through its public entry points.

Every case is one call that a serving program makes on an ``Engine`` it keeps:

* ``call="layer"``: one ``layer_step`` of a large batch in the middle of the
  model (plain launches, every per-token output asked for), the unit that a
  program with its own layer loop runs;
* ``call="forward"``: ``forward`` over a few layers with graph replay on a
  stream of its own, which is how small batches are served;
* ``call="host"``: ``forward_host`` on pinned host buffers.

Shapes are the repository's own model families (``workload.CONFIGS``): a
Switch-Base-8E-shaped layer (top-1 ReLU, 64-class exit head), a
Qwen-MoE-A2.7B-shaped one (60 experts, top-4 SwiGLU, shared expert) and a
Mixtral-8x7B-shaped one (top-2 of 8 large SwiGLU experts), with the attention
sublayer or the exit prediction where a case says so.  A few layers stand for
the model's 12 to 32: a layer's work does not depend on the number of others.
A pass starts from the same token state each time (a device copy, as a program
does that hands new tokens to buffers it keeps).
"""
import math

import numpy as np
import torch

from paper_2608_00573_gb300 import binding as B
from paper_2608_00573_gb300 import workload as W

# Calibrated thresholds and exit biases are those of the family's layers from
# this depth on, where tokens skip and exit.
DEPTH = {"switch": 4, "qwen": 8, "mixtral": 18, "mixtral_decode": 18}
CENTROIDS = 64


def _case(name, family, call, tokens, layers, attention=False, prediction=False, budget=0.02):
    c = dict(family=family, call=call, tokens=tokens, layers=layers, attention=attention,
             prediction=prediction, budget=budget)
    return dict(c, name=name) if name else c


def listed():
    return [
        # The smallest call: one 64-token batch through the smallest model, where latency and launches count.
        _case("switch_forward_64", "switch", "forward", 64, 4),
        # The same model fed from host memory: an odd batch, copied in and out inside the call.
        _case("switch_host_777", "switch", "host", 777, 4),
        # A full batch of the small model: short GEMMs between small kernels.
        _case("switch_layer_4096", "switch", "layer", 4096, 3),
        # Decode of eight sequences on many small experts and a shared expert.
        _case("qwen_forward_8", "qwen", "forward", 8, 4),
        # A ragged medium batch (one long prompt): a few rows per expert.
        _case("qwen_forward_333", "qwen", "forward", 333, 4),
        # A full prefill batch of the many-expert model, ragged groups of about 500 rows.
        _case("qwen_layer_8192", "qwen", "layer", 8192, 3),
        # Decode of one sequence: two experts' weights a layer.
        _case("mixtral_forward_1", "mixtral_decode", "forward", 1, 6),
        # Decode of an odd number of sequences: nearly every expert's weights stream once.
        _case("mixtral_forward_113", "mixtral_decode", "forward", 113, 4),
        # An odd medium prefill with exit-point prediction against 64 centroids.
        _case("mixtral_layer_1500_predict", "mixtral", "layer", 1500, 3, prediction=True),
        # The largest call: a full prefill batch.
        _case("mixtral_layer_16384", "mixtral", "layer", 16384, 3),
        # Prefill of one user's 128 tokens through whole transformer blocks.
        _case("mixtral_block_128", "mixtral", "forward", 128, 4, attention=True),
        # A batched prefill through a whole block, its last sequence ragged.
        _case("mixtral_block_4200", "mixtral", "layer", 4200, 3, attention=True),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    family = rng.choice(["switch", "qwen", "mixtral"])
    call = rng.choice(["layer", "forward", "layer", "forward", "host"])
    attention = rng.random() < 0.25
    prediction = rng.random() < 0.25
    if call == "layer":     # prefill batches
        top = {"switch": 8192, "qwen": 8192, "mixtral": 16384}[family]
        if attention or prediction:
            top //= 2
        return _case(None, family, call, _log_int(rng, 256, top), 3, attention, prediction)
    if call == "host":
        return _case(None, "switch", call, _log_int(rng, 32, 1024), rng.randint(3, 6))
    if family == "mixtral" and not attention and rng.random() < 0.7:
        return _case(None, "mixtral_decode", call, _log_int(rng, 1, 256), rng.randint(3, 8), False, prediction,
                     rng.choice([0.005, 0.02, 0.05]))
    return _case(None, family, call, _log_int(rng, 1, 512), rng.randint(3, 6), attention, prediction)


def _config(case, seed):
    """The workload of a case: a slice of its family's layers, every draw by the seed."""
    fam = case["family"]
    cfg = W.CONFIGS[fam].replace(N=case["layers"], T=case["tokens"], budget=case["budget"], seed=int(seed),
                                 n_centroids=CENTROIDS if case["prediction"] else 0)
    if case["prediction"]:
        cfg = cfg.replace(exit_peak=1.5 if cfg.N <= 3 else 0.7 * cfg.N, exit_width=1.0)
    if case["attention"]:
        cfg = W.with_attention(cfg)
    cal = W.load_calibration(fam)
    a = DEPTH[fam]
    cal = {k: cal[k][a:a + cfg.N] for k in ("theta", "exit_bias")}
    return cfg, cal


FIELDS = (("hidden", torch.bfloat16), ("s", torch.uint8), ("Dhat", torch.float32), ("Dbar", torch.float32),
          ("pJ", torch.float32), ("alive", torch.uint8), ("last_exec", torch.uint8), ("xi_last", torch.float32),
          ("exit_layer", torch.int16))


def _views(flat, T, d):
    """The token fields as views of one byte buffer, each at a 256-byte boundary."""
    out, at = {}, 0
    for name, dt in FIELDS:
        n = T * (d if name == "hidden" else 1)
        size = n * torch.empty((), dtype=dt).element_size()
        if flat is not None:
            v = flat[at:at + size].view(dt)
            out[name] = v.view(T, d) if name == "hidden" else v
        at += (size + 255) // 256 * 256
    return out, at


def _tokens(case, cfg, seed):
    """Token states on the GPU: new tokens for a forward, tokens in the middle of
    the model (some of them gone, skipped or partly through their budget) for a
    layer."""
    T, M = case["tokens"], cfg.M
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 31 + 7)
    _, size = _views(None, T, cfg.d)
    flat = torch.zeros(size, dtype=torch.uint8, device="cuda")
    v, _ = _views(flat, T, cfg.d)

    def u():
        return torch.rand(T, generator=g, device="cuda")

    v["hidden"].normal_(0.0, 1.0, generator=g)
    zipf = 1.0 / torch.arange(1, M + 1, device="cuda", dtype=torch.float64)      # users by access server
    users = torch.multinomial(zipf, (T + 127) // 128, replacement=True, generator=g)
    v["s"].copy_(users.repeat_interleave(128)[:T])
    v["Dbar"].fill_(cfg.budget)
    v["pJ"].fill_(cfg.p_J)
    v["alive"].fill_(1)
    v["xi_last"].fill_(-1.0)
    v["exit_layer"].fill_(cfg.N)
    if case["call"] == "layer":
        gone = u() < 0.08
        v["alive"].masked_fill_(gone, 0)
        v["exit_layer"].masked_fill_(gone, 0)
        v["last_exec"].copy_(u() < 0.88)
        v["Dhat"].copy_(cfg.budget * 0.9 * u() * (u() < 0.6))
        v["s"].copy_(torch.where(u() < 0.5, v["s"], torch.randint(0, M, (T,), generator=g, device="cuda").to(torch.uint8)))
    return flat


def _model(case, seed):
    cfg, cal = _config(case, seed)
    small = W.make_small_weights(cfg, calib=cal)
    tables = W.make_tables(cfg, small["W_r"], calib=cal)
    return cfg, small, tables, W.make_expert_weights_device(cfg)


def prepare(case, seed):
    cfg, small, tables, experts = _model(case, seed)
    T, call = case["tokens"], case["call"]
    eng = B.Engine(cfg, tables, small, experts, T_max=T, graphs=call != "layer")
    init = _tokens(case, cfg, seed)
    st = dict(case=case, eng=eng, stream=torch.cuda.Stream() if call != "layer" else torch.cuda.current_stream())
    if call == "host":
        init = init.cpu().pin_memory()
        work = torch.empty_like(init, pin_memory=True)
    else:
        work = torch.empty_like(init)
    st.update(init=init, work=work, tok=_views(work, T, cfg.d)[0])
    if call == "layer":
        st["out"] = eng.alloc_layer_out(T)
        st["out"].update(perm=None, group_off=None, h_attn=None)     # a layer loop has no use for these
        if not cfg.n_centroids:
            st["out"]["lhat"] = None
    return st


def run(state):
    eng, tok, call = state["eng"], state["tok"], state["case"]["call"]
    if call == "layer":
        state["work"].copy_(state["init"])
        eng.layer_step(1, tok, out=state["out"])
        return {"tok": _result(tok), "out": {k: v for k, v in state["out"].items() if v is not None}}
    with torch.cuda.stream(state["stream"]):
        state["work"].copy_(state["init"])
        if call == "host":
            eng.forward_host(tok, stream=state["stream"])
        else:
            eng.forward(tok, stream=state["stream"])
    return {"tok": _result(tok)}


def _result(tok):
    return {k: v for k, v in tok.items() if k not in ("Dbar", "pJ")}      # those two are read only


# ------------------------------------------------------------------ work

def work(case):
    """One pass with the expected numbers of executed pairs and of experts that get any."""
    cfg, _ = _config(case, 0)
    layer = case["call"] == "layer"
    n, live = (1 if layer else cfg.N), case["tokens"] * (0.92 if layer else 1.0)
    rows = live * 0.86 if layer else live * 0.9      # executed: neither skipped nor exited
    pairs = rows * cfg.k
    pop = np.arange(1, cfg.E + 1, dtype=np.float64) ** -cfg.zipf_s
    pop /= pop.sum()
    # Tokens of one user start on one server and prefer what is deployed there
    # (substitutes included): with one user about half as many experts get work
    # as routing alone would touch, and nearly all of them from about five on.
    users = (case["tokens"] + 127) // 128
    touched = min(float(np.sum(1.0 - (1.0 - pop) ** pairs)), pairs) * min(1.0, 0.55 + 0.12 * (users - 1))
    mats = (cfg.n13 + 1) * cfg.F * cfg.d
    n_out = cfg.E + cfg.C + cfg.n_centroids
    flops = 2.0 * pairs * mats + 2.0 * live * n_out * cfg.d
    byts = 2.0 * touched * mats + 2.0 * n_out * cfg.d + 2 * 2.0 * live * cfg.d + 32.0 * live
    if cfg.F_sh:
        flops += 2.0 * live * 3 * cfg.F_sh * cfg.d
        byts += 2.0 * 3 * cfg.F_sh * cfg.d
    if cfg.attn_heads:
        hd = cfg.attn_heads * cfg.head_dim
        flops += 2.0 * case["tokens"] * cfg.d * (cfg.n_qkv + hd) + 4.0 * hd * case["tokens"] * min(64, case["tokens"])
        byts += 2.0 * cfg.d * (cfg.n_qkv + hd)
    if case["call"] == "host":
        byts += 2.0 * (2.0 * cfg.d + 19) * live
    return {"bytes": n * byts, "flops": n * flops}


def tolerance(case):
    """Measured against exact(): one MoE layer's hidden states are 1.6e-3 to
    2.0e-3 off (bf16 activations and expert outputs, a bf16 result), and no
    decision differs; four times that.  Where a bf16 state is rounded again before
    a later decision (several layers, or an attention sublayer in front of the
    router), a last-bit change of it can move a token across a threshold, and its
    row with it: 4e-3 to 6e-2 off, a token in a hundred decided otherwise."""
    if case["call"] == "layer" and not case["attention"]:
        return {"rel": 7e-3, "max": 0.1, "differ": 1e-3}
    return {"rel": 3e-2, "max": 0.9, "differ": 1e-2}


# ------------------------------------------------------------------ exact

def _bf(x):
    return x.to(torch.bfloat16).to(torch.float64)


def exact(case, seed):
    """The layer's definition in 64 bits; bf16 where a stored state or an operand
    is bf16 by the entry point's contract (hidden states, normalised inputs, q, k
    and v), nowhere else."""
    w = work(case)["flops"]
    if w > 1.5e13:
        return None
    cfg, small, tab, ex = _model(case, seed)
    T, E, K, M, d, N = case["tokens"], cfg.E, cfg.k, cfg.M, cfg.d, cfg.N
    dev = "cuda"
    f64 = torch.float64

    def dd(a):
        return torch.as_tensor(np.asarray(a, dtype=np.float64), device=dev)

    def wt(name, l):
        return dd(W.bf16_bits_to_f32(small[name][l]))

    v, _ = _views(_tokens(case, cfg, seed), T, d)
    h = v["hidden"].to(f64)
    s = v["s"].long()
    Dh, Db, pJ = v["Dhat"].to(f64), v["Dbar"].to(f64), v["pJ"].to(f64)
    alive, last = v["alive"].bool(), v["last_exec"].bool()
    xi_last, exit_layer = v["xi_last"].to(f64), v["exit_layer"].long()
    trans, comp, P = dd(tab["trans"]), dd(tab["comp"]), dd(tab["P"]) if N > 1 else None
    place = torch.as_tensor(tab["place"].astype(np.int64), device=dev)
    srv = torch.arange(M, device=dev)
    inf = float("inf")

    # Candidates of layer l: feasible[r, k, m] and loss Q[r, k] (the exact expert, then the n_sub most similar).
    def candidates(l):
        sim = dd(tab["sim"][l])
        off = sim.clone()
        off.fill_diagonal_(-inf)
        off = torch.where(off >= float(tab["sub_thresh"][l]), off, torch.full_like(off, -inf))
        ok = torch.eye(E, dtype=torch.bool, device=dev)
        order = torch.sort(off, dim=1, descending=True, stable=True)
        for j in range(min(cfg.n_sub, E - 1)):
            got = order.values[:, j] > -inf
            ok[torch.arange(E, device=dev)[got], order.indices[got, j]] = True
        Q = cfg.phi_beta * (1.0 - sim) / 2.0
        Q.fill_diagonal_(0.0)
        deployed = ((place[l][:, None] >> srv[None, :]) & 1).bool()          # [k, m]
        return ok[:, :, None] & deployed[None], Q

    move = cfg.omega_T * trans * (1 - torch.eye(M, device=dev, dtype=f64)) / tab["d_ref"]     # [from, to]

    # Cost-to-go tables Phi_l(m, k) for budgets R: [n, M, E].
    def lookahead(l, R, budget, cap):
        top = min(cfg.H - 1, N - 1 - l, cap)
        phi = torch.zeros(len(R), M, E, dtype=f64, device=dev)
        for j in range(top, 0, -1):
            lp = l + j
            ok, Q = candidates(lp)
            V = torch.full((len(R), M, E), inf, dtype=f64, device=dev)
            local = torch.zeros(len(R), M, E, dtype=torch.bool, device=dev)
            for k in range(E):           # executed expert k, for every target r that admits it
                base = move + cfg.omega_T * comp[lp][None, :] / tab["d_ref"]            # [m, m']
                val = base[None] + phi[:, None, :, k]                                    # [n, m, m']
                for r in torch.nonzero(ok[:, k].any(1)).flatten().tolist():
                    fit = (Q[r, k] <= R)[:, None, None] & ok[r, k][None, None, :]
                    c = torch.where(fit, val + cfg.omega_D * Q[r, k] / budget, torch.full_like(val, inf))
                    V[:, :, r] = torch.minimum(V[:, :, r], c.min(2).values)
                    local[:, :, r] |= (Q[r, k] <= R)[:, None] & ok[r, k][None, :]
            eps = float(tab["eps"][lp])
            skip = cfg.omega_D * eps / budget + phi
            V = torch.where(~local & (eps <= R)[:, None, None], torch.minimum(V, skip), V)
            phi = torch.einsum("kq,nmq->nmk", P[lp - 1], V)
        return phi

    def attention(l, x):
        Hq, Hk, D, S = cfg.attn_heads, cfg.attn_kv_heads, cfg.head_dim, cfg.attn_seq
        a = _bf(x / torch.sqrt((x * x).mean(1, keepdim=True) + cfg.norm_eps) * wt("W_attn_norm", l))
        z = a @ ex["W_qkv"][l].to(f64).T
        pos = torch.arange(T, device=dev) % S
        ang = pos[:, None].to(f64) * float(cfg.rope_theta) ** (-2.0 * torch.arange(D // 2, device=dev, dtype=f64) / D)
        c, sn = torch.cos(ang)[:, None], torch.sin(ang)[:, None]
        qk = z[:, :(Hq + Hk) * D].view(T, Hq + Hk, D)
        lo, hi = qk[..., :D // 2], qk[..., D // 2:]
        qk = _bf(torch.cat([lo * c - hi * sn, hi * c + lo * sn], -1))
        val = _bf(z[:, (Hq + Hk) * D:]).view(T, Hk, D).repeat_interleave(Hq // Hk, 1)
        key = qk[:, Hq:].repeat_interleave(Hq // Hk, 1)
        o = torch.empty(T, Hq, D, dtype=f64, device=dev)
        for t in range(0, T, S):
            n = min(S, T - t)
            sc = torch.einsum("qhd,khd->hqk", qk[t:t + n, :Hq], key[t:t + n]) / math.sqrt(D)
            sc = sc.masked_fill(torch.ones(n, n, dtype=torch.bool, device=dev).triu(1), -inf)
            o[t:t + n] = torch.einsum("hqk,khd->qhd", torch.softmax(sc, -1), val[t:t + n])
        return _bf(x + o.reshape(T, Hq * D) @ ex["W_o"][l].to(f64).T)

    def ffn(x, w13, w2, act):
        if act == W.ACT_SWIGLU:
            g = w13.view(-1, 2, W.GATE_UP_GROUP, d)
            gate = x @ g[:, 0].reshape(-1, d).to(f64).T
            a = torch.nn.functional.silu(gate) * (x @ g[:, 1].reshape(-1, d).to(f64).T)
        else:
            a = torch.relu(x @ w13.to(f64).T)
        return a @ w2.to(f64).T

    out = {}
    for l in ([1] if case["call"] == "layer" else range(N)):
        h_in = h
        hm = attention(l, h) if cfg.attn_heads else h
        r = 1.0 / torch.sqrt((hm * hm).mean(1, keepdim=True) + cfg.norm_eps)
        xn = hm * r * wt("W_norm", l)
        z = xn @ wt("W_r", l).T + dd(small["b_r"][l])
        p = torch.softmax(z, 1)
        top = torch.sort(z, dim=1, descending=True, stable=True).indices[:, :K]
        g = p.gather(1, top)
        I = g.sum(1)
        xi = torch.full((T,), -1.0, dtype=f64, device=dev)
        if l > 0:
            rx = 1.0 / torch.sqrt((h_in * h_in).mean(1, keepdim=True) + cfg.norm_eps)
            x = (h_in * rx) @ wt("W_x", l - 1).T + dd(small["b_x"][l - 1])
            conf = torch.sigmoid(x[:, 0]) if cfg.C == 1 else torch.softmax(x, 1).max(1).values
            xi = torch.where(last & alive, conf, xi)
        cap = torch.full((T,), N, dtype=torch.long, device=dev)
        lhat = cap.clone()
        if cfg.n_centroids:
            ce = wt("centroids", l)
            near = (h_in @ ce.T / ce.norm(dim=1)).argmax(1)
            lhat = torch.floor(dd(small["centroid_exit"][l]) + 0.5).long()[near]
            cap = (lhat - 1 - l).clamp(min=0)
        # Every token's Phi: one table for each interval of R between thresholds and each cap.
        R = Db - Dh
        depth = min(cfg.H - 1, N - 1 - l)
        thr = [dd([float(e) for e in tab["eps"][l + 1:l + 1 + depth]])]
        thr += [candidates(l + j)[1].flatten() for j in range(1, depth + 1)]
        iv = torch.bucketize(R, torch.unique(torch.cat(thr)), right=True)
        phi = torch.zeros(T, M, E, dtype=f64, device=dev)
        for cp in torch.unique(cap.clamp(max=depth)).tolist():
            at = torch.nonzero(cap.clamp(max=depth) == cp).flatten()
            ids, inv = torch.unique(iv[at], return_inverse=True)
            rep = torch.zeros(len(ids), dtype=f64, device=dev).scatter_reduce(0, inv, R[at], "amax", include_self=False)
            for b in range(0, len(ids), 64):
                tb = lookahead(l, rep[b:b + 64], float(case["budget"]), cp)
                sel = (inv >= b) & (inv < b + 64)
                phi[at[sel]] = tb[inv[sel] - b]
        ok, Q = candidates(l)
        Gamma = torch.zeros(T, dtype=f64, device=dev)
        lam = float(tab["lam"][l]) * I
        run_D, total, esel, msel = Dh.clone(), torch.zeros(T, dtype=f64, device=dev), [], []
        away = 1 - torch.eye(M, device=dev, dtype=f64)
        for j in range(K):
            t = top[:, j]
            q = Q[t]                                                   # [T, k]
            fit0 = ok[t] & (Dh[:, None] + q <= Db[:, None])[:, :, None]  # [T, k, m]
            hop = (trans * away)[s][:, None, :].expand(-1, E, -1)
            Gamma += torch.where(fit0, hop, torch.full_like(hop, inf)).flatten(1).min(1).values
            fit = fit0 & (run_D[:, None] + q <= Db[:, None])[:, :, None]
            cost = (move[s] + cfg.omega_T * comp[l] / tab["d_ref"])[:, None, :] + (cfg.omega_D * q / Db[:, None])[:, :, None]
            if j == 0:
                cost = cost + phi.transpose(1, 2)
            cost = torch.where(fit, cost, torch.full_like(cost, inf))
            # ties go to the exact expert, then to the lower index
            rank = torch.cat([cost.gather(1, t[:, None, None].expand(-1, 1, M)), cost], 1).flatten(1)
            best = rank.min(1)
            i = best.indices
            e = torch.where(i < M, t, torch.div(i, M, rounding_mode="floor") - 1)
            esel.append(e)
            msel.append(i % M)
            run_D = run_D + q.gather(1, e[:, None])[:, 0]
            total = total + best.values
        skip_ok = (Gamma > 0) & (I <= float(tab["theta"][l])) & (Dh + lam <= Db)
        skip_cost = cfg.omega_D * lam / Db + phi[torch.arange(T, device=dev), s, top[:, 0]]
        action = torch.where(skip_ok & (skip_cost < total), 1, 0)
        best = torch.where(action == 1, skip_cost, total)
        action = torch.where((xi >= pJ) & last & (best > 0) & (l > 0), 2, action)
        action = torch.where(alive, action, 3)
        did, skip, left = action == 0, action == 1, action == 2
        # expert FFNs on the executed pairs, combined in slot order
        acc = hm.clone()
        xb = _bf(xn)
        gw = g / g.sum(1, keepdim=True) if cfg.renorm_topk else g
        for e in range(E):
            rows = torch.zeros(T, dtype=f64, device=dev)
            hit = torch.zeros(T, dtype=torch.bool, device=dev)
            for j in range(K):
                m = did & (esel[j] == e)
                rows = rows + torch.where(m, gw[:, j], torch.zeros_like(rows))
                hit |= m
            at = torch.nonzero(hit).flatten()
            if len(at):
                acc[at] += rows[at][:, None] * ffn(xb[at], ex["W13"][l, e], ex["W2"][l, e], cfg.act)
        at = torch.nonzero(did | skip).flatten()
        if cfg.F_sh and len(at):
            acc[at] += ffn(xb[at], ex["W13_sh"][l], ex["W2_sh"][l], W.ACT_SWIGLU)
        h = torch.where((did | skip)[:, None], acc, h_in)
        off = torch.full((T, K), 255, dtype=torch.long, device=dev)
        out = {"topk_idx": torch.where(alive[:, None], top, -1).flatten(), "topk_g": torch.where(alive[:, None], g, 0.0).flatten(),
               "I": torch.where(alive, I, 0.0), "xi": xi, "action": action,
               "exp_sel": torch.where(did[:, None], torch.stack(esel, 1), off).flatten(),
               "srv_sel": torch.where(did[:, None], torch.stack(msel, 1), off).flatten()}
        if cfg.n_centroids:
            out["lhat"] = torch.where(alive, lhat, -1)
        s = torch.where(did, msel[0], s)
        Dh = torch.where(did, run_D, torch.where(skip, Dh + lam, Dh))
        xi_last = torch.where(xi >= 0, xi, xi_last)
        last = torch.where(did, True, torch.where(skip, False, last))
        exit_layer = torch.where(left, l, exit_layer)
        alive = alive & ~left
        if case["call"] != "layer" and l + 1 < N:
            h = _bf(h)
    tok = {"hidden": h, "s": s, "Dhat": Dh, "alive": alive.long(), "last_exec": last.long(), "xi_last": xi_last,
           "exit_layer": exit_layer}
    return {"tok": tok, "out": out} if case["call"] == "layer" else {"tok": tok}
