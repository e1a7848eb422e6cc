"""Performance cases of the DiG token mixer: what a program that uses this package has it do.

The cases are forward and training passes of one mixer block through the public entry points, over the
image sizes, model sizes, batch sizes and storage types of the repository's workloads (`inputs.CONFIGS`:
grids of 16 x 16 to 128 x 128 tokens, heads of 64 channels for the S and B sizes and of 72 for XL), plus the
operator variants the package offers: fp32 storage, the full gate, the sum over four scan orders and the
recurrence cut into pieces.

`op` of a case:
  infer        gate transform, GLA forward with the output gate, SREM conv
  bands        the same operator row band by row band of an image, the state handed from band to band
  train        the block's forward pass with what it keeps for the backward pass, then the backward pass:
               conv, output gate and GLA gradients, each fed by the one before
  full_gate    forward and backward with the value-channel gate beside the key-channel gate
  four_scans   forward and backward of the sum over all four scan orders
"""
import math

import torch

from paper_2405_18428_b200 import dig

_EPS = 1e-5


def _case(name, op, dtype, B, H, grid_h, grid_w, d, direction=0, chunk=64, tau=16.0, tau2=16.0, bands=1):
    c = dict(op=op, dtype=dtype, B=B, H=H, grid_h=grid_h, grid_w=grid_w, d=d, direction=direction, chunk=chunk, tau=tau,
             tau2=tau2, bands=bands)
    return c if name is None else dict(name=name, **c)


def listed():
    return [
        # one 256 x 256 image through one S-size block: the smallest call, launches and latency count
        _case("infer_256px_s", "infer", "bf16", 1, 6, 16, 16, 64),
        # the same in fp32 storage, as for reference results and small checks (workload C1)
        _case("infer_256px_s_f32", "infer", "f32", 1, 6, 16, 16, 64),
        # a 1792 x 1792 image (workload C4) fed in four row bands with the state handed over
        _case("bands_1792px_s", "bands", "bf16", 1, 6, 112, 112, 64, bands=4),
        # one 2048 x 2048 image through an XL block, a reversed column scan (workload C5)
        _case("infer_2048px_xl", "infer", "bf16", 1, 16, 128, 128, 72, direction=3),
        # training at 256 x 256: many short sequences
        _case("train_256px_s_batch", "train", "bf16", 128, 6, 16, 16, 64, direction=1),
        # training at 512 x 512 (workload C2), a column scan
        _case("train_512px_s", "train", "bf16", 8, 6, 32, 32, 64, direction=2),
        # training at 1024 x 1024, B size, heads of different gate temperature (workload C3)
        _case("train_1024px_b", "train", "bf16", 4, 12, 64, 64, 64, tau2=4.0),
        # training at 2048 x 2048, XL size (workload C5): the largest
        _case("train_2048px_xl", "train", "bf16", 1, 16, 128, 128, 72, direction=1),
        # an odd grid whose sequences end inside a tile, chunks of 32 tokens, heads of 72
        _case("train_ragged_xl", "train", "bf16", 3, 16, 37, 53, 72, direction=3, chunk=32),
        # training in fp32 storage
        _case("train_512px_s_f32", "train", "f32", 2, 6, 32, 32, 64, direction=2),
        # training with the paper's full gate
        _case("full_gate_512px_s", "full_gate", "bf16", 8, 6, 32, 32, 64, tau2=4.0),
        # training with four scan directions summed (the paper's comparison of scanning strategies)
        _case("four_scans_512px_s", "four_scans", "bf16", 8, 6, 32, 32, 64),
    ]


# The largest listed case's work in output elements of its GLA gradients; a drawn case stays at or below it.
_MOST = 128 * 128 * 16 * 72


def draw(rng):
    """One more case: an op with its share of use, a model size, then grid sides and batch spread over their
    logarithm."""
    op = rng.choices(["infer", "train", "bands", "full_gate", "four_scans"], [30, 45, 8, 9, 8])[0]
    dtype = "f32" if op in ("infer", "train", "full_gate") and rng.random() < 0.2 else "bf16"
    H, d = rng.choice([(6, 64), (12, 64), (16, 64), (16, 72)])
    slow = dtype == "f32" or op in ("full_gate", "four_scans")
    most = _MOST // (8 if slow else 1)
    side = lambda lo, hi: max(lo, min(hi, round(math.exp(rng.uniform(math.log(lo), math.log(hi))))))
    while True:
        gh = side(8, 64 if slow else 128)
        gw = gh if rng.random() < 0.4 else side(max(8, gh // 2), min(64 if slow else 128, 2 * gh))
        room = most // (gh * gw * H * d)
        if room >= 1:
            break
    B = 1 if op == "bands" or (op == "infer" and rng.random() < 0.5) else side(1, min(room, 128))
    return _case(None, op, dtype, B, H, gh, gw, d, direction=0 if op == "bands" else rng.randrange(4),
                 chunk=rng.choice([64, 64, 64, 32]), tau=16.0, tau2=rng.choice([16.0, 16.0, 4.0]),
                 bands=min(gh, rng.choice([2, 3, 4])) if op == "bands" else 1)


def prepare(case, seed):
    B, H, d, gh, gw, op = (case[k] for k in ("B", "H", "d", "grid_h", "grid_w", "op"))
    L, D = gh * gw, H * d
    gen = torch.Generator(device="cuda").manual_seed(seed)
    st = torch.float32 if case["dtype"] == "f32" else torch.bfloat16

    def normal(*shape, scale=1.0, dtype=st):
        return (torch.randn(shape, generator=gen, device="cuda") * scale).to(dtype)

    # query and key are N(0, 1) each and correlated within a token, as two projections of one token are.  With
    # independent ones q.k of a sequence's first token is close to 0 now and then, and the layer norm of that
    # token's output, (q.k) v, would have no significant digits in any implementation.
    q = torch.randn((B, L, H, d), generator=gen, device="cuda")
    k = (0.7 * q + math.sqrt(1 - 0.7 ** 2) * normal(B, L, H, d, dtype=torch.float32)).to(st)
    s = dict(case=case, q=q.to(st), k=k, v=normal(B, L, H, d), g=normal(B, L, H, d),
             tau=[case["tau"] if h % 2 == 0 else case["tau2"] for h in range(H)])
    if op in ("infer", "bands", "train"):
        s["r"] = normal(B, L, H, d)
        s["ln_w"] = 1 + normal(d, scale=0.1, dtype=torch.float32)
        s["ln_b"] = normal(d, scale=0.1, dtype=torch.float32)
        s["w"] = normal(3, 3, D, scale=1 / 3)                   # variance 1/9
        s["bias"] = normal(D, scale=0.1)
    if op == "train":
        s["dy"] = normal(B, L, D)
    if op in ("full_gate", "four_scans"):
        s["dO"] = normal(B, L, H, d)
    if op == "full_gate":
        s["gv"] = normal(B, L, H, d)
        s["tau_v"] = [8.0] * H                                  # the value gate decays at its own temperature
    if op == "bands":
        # a program that feeds bands holds each band as tensors of its own
        n, b = case["bands"], []
        cut = [gh * i // n for i in range(n + 1)]
        for lo, hi in zip(cut, cut[1:]):
            b.append((hi - lo, [s[x][:, lo * gw:hi * gw].contiguous() for x in ("q", "k", "v", "g", "r")]))
        for x in ("q", "k", "v", "g", "r"):
            del s[x]
        s["parts"] = b
    return s


def _infer(c, s):
    gh, gw, ch, di = c["grid_h"], c["grid_w"], c["chunk"], c["direction"]
    gate = dig.dig_gate_logsigmoid(s["g"], s["tau"])
    _, z = dig.dig_gla_fwd_outgate(s["q"], s["k"], s["v"], gate, s["r"], gh, gw, ch, di, ln_w=s["ln_w"], ln_b=s["ln_b"],
                                   eps=_EPS, want_out=False)
    return dig.dig_srem_dwconv(z.view(c["B"], gh * gw, -1), s["w"], s["bias"], gh, gw, di)


def _bands(c, s):
    state, ys = None, []
    for rows, (q, k, v, g, r) in s["parts"]:
        gate = dig.dig_gate_logsigmoid(g, s["tau"])
        o, state = dig.dig_gla_fwd_state(q, k, v, gate, state, rows, c["grid_w"], c["chunk"], 0)
        ys.append(dig.dig_gla_outgate_fwd(o, r, s["ln_w"], s["ln_b"], _EPS))
    return ys, state


def _train(c, s):
    gh, gw, ch, di = c["grid_h"], c["grid_w"], c["chunk"], c["direction"]
    flat = (c["B"], gh * gw, c["H"] * c["d"])
    q, k, v, r = s["q"], s["k"], s["v"], s["r"]
    gate = dig.dig_gate_logsigmoid(s["g"], s["tau"])
    o = dig.dig_gla_fwd(q, k, v, gate, gh, gw, ch, di)
    z = dig.dig_gla_outgate_fwd(o, r, s["ln_w"], s["ln_b"], _EPS)
    y = dig.dig_srem_dwconv(z.view(flat), s["w"], s["bias"], gh, gw, di)
    dz, dw, dbias = dig.dig_srem_dwconv_bwd(z.view(flat), s["w"], s["dy"], gh, gw, di)
    d_o, d_r, dln_w, dln_b = dig.dig_gla_outgate_bwd(o, r, dz.view(o.shape), s["ln_w"], s["ln_b"], _EPS)
    grads = dig.dig_gla_bwd(q, k, v, gate, d_o, gh, gw, ch, di)
    return y, grads, d_r, dln_w, dln_b, dw, dbias


def _full_gate(c, s):
    gh, gw, ch, di = c["grid_h"], c["grid_w"], c["chunk"], c["direction"]
    gate = dig.dig_gate_logsigmoid(s["g"], s["tau"])
    bgate = dig.dig_gate_logsigmoid(s["gv"], s["tau_v"])
    out = dig.dig_gla_fwd_beta(s["q"], s["k"], s["v"], gate, bgate, gh, gw, ch, di)
    return out, dig.dig_gla_bwd_beta(s["q"], s["k"], s["v"], gate, bgate, s["dO"], gh, gw, ch, di)


def _four_scans(c, s):
    gh, gw, ch = c["grid_h"], c["grid_w"], c["chunk"]
    gate = dig.dig_gate_logsigmoid(s["g"], s["tau"])
    out = dig.dig_gla_fwd_multi(s["q"], s["k"], s["v"], gate, gh, gw, range(4), ch)
    return out, dig.dig_gla_bwd_multi(s["q"], s["k"], s["v"], gate, s["dO"], gh, gw, range(4), ch)


_RUN = {"infer": _infer, "bands": _bands, "train": _train, "full_gate": _full_gate, "four_scans": _four_scans}


def run(state):
    c = state["case"]
    return _RUN[c["op"]](c, state)


def work(case):
    """Bytes: what the block reads and writes at its ends plus the gates and, in training, what the forward
    pass has to keep (written once, read once); filters, affine weights and states are left out as small.
    Flops: the recurrence token by token (the state's decay and update and the readout, per element of the
    state), twice that and the state again for its derivative; the conv and its derivative."""
    n = case["B"] * case["grid_h"] * case["grid_w"] * case["H"] * case["d"]
    w = 4 if case["dtype"] == "f32" else 2
    fwd = 5 * case["d"] * n
    bwd = 13 * case["d"] * n
    op = case["op"]
    if op in ("infer", "bands"):
        # q k v g r in, y out
        return {"bytes": n * 6 * w, "flops": fwd + (18 * n if op == "infer" else 0)}
    if op == "train":
        # in: q k v g r dy; out: y dq dk dv dr, fp32 dgate; kept and read back: the gate, o, z (and q k v r read again)
        return {"bytes": n * (6 * w + 5 * w + 4 + 2 * (4 + 2 * w) + 4 * w), "flops": fwd + bwd + 54 * n}
    if op == "full_gate":
        # in: q k v dO and two gate logits; out: out dq dk dv and two fp32 gate gradients
        return {"bytes": n * (6 * w + 4 * w + 8), "flops": (fwd + bwd) * 6 // 5}
    return {"bytes": n * (5 * w + 4 * w + 4), "flops": 4 * (fwd + bwd)}


def tolerance(case):
    """About four times the largest relative error seen against the same chain in fp64 (token-by-token
    recurrence): 3.1e-3 with bf16 storage, 4.4e-7 in fp32 storage (the gate gradient, a running sum, grows with
    the length: 1e-6), 2.8e-5 for the full gate in fp32 storage."""
    if case["dtype"] == "bf16":
        return {"rel": 1.2e-2}
    return {"rel": 1e-4 if case["op"] == "full_gate" else 4e-6}
