"""What the performance of this framework is measured on: the calls that its users make, each
through the public entry points of paper_2410_05911_gb300.aecct.

Four entry points, each a "kind" of case:

  decode     Decoder.decode on received words that are already on the GPU (a receiver chain or a
             simulation loop on the device).
  host       Decoder.decode_host: words in host memory, decoded words back in host memory.
  ternarize  aap_ternarize: the weight quantiser that training applies to every weight tensor in
             its forward pass, and that an export applies once to a trained model.
  spe        spe_table: the spectral positional encoding of a new code's Tanner graph.

Codes are BCH(31,16), BCH(63,36), Polar(64,32) and (3,6)-regular LDPC codes, models have d in
{32, 64, 128}, 1 to 10 blocks and random weights of a trained model's shapes; batches run from one
word (latency) to the benchmark's 262,144 (throughput).  "variant" picks the model's options:
"aap" (ternary linears, HPSA, ReLU), "gelu" (the same with GELU), "fp" (full-precision linears on
bf16 tensor cores, HPSA, ReLU) and "ecct" (full-precision linears, the code-aware mask on every
head, GELU: the ECCT baseline).
"""
import math

import numpy as np
import torch

from paper_2410_05911_gb300 import aecct, inputs

HEADS = 8


def listed():
    return [
        # one received word of the smallest model: the latency of a single call
        dict(name="bch31_16_one", kind="decode", code="bch31_16", d=32, layers=2, variant="aap", batch=1),
        # the smallest benchmark configuration: a short batch in a real-time loop
        dict(name="bch31_16", kind="decode", code="bch31_16", d=32, layers=2, variant="aap", batch=1024),
        # the deepest model on fewer words than the GPU holds at once: a lightly loaded receiver
        dict(name="bch63_36_few", kind="decode", code="bch63_36", d=128, layers=10, variant="aap", batch=37),
        # the throughput benchmarks of the four larger codes: bulk decoding or a BER simulation
        dict(name="polar64_32", kind="decode", code="polar64_32", d=64, layers=6, variant="aap", batch=65536),
        dict(name="bch63_36", kind="decode", code="bch63_36", d=128, layers=10, variant="aap", batch=262144),
        dict(name="ldpc128_64", kind="decode", code="ldpc128_64", d=128, layers=6, variant="aap", batch=131072),
        dict(name="ldpc384_192", kind="decode", code="ldpc384_192", d=128, layers=6, variant="aap", batch=16384),
        # a code of more than 128 tokens on the middle width, an odd batch
        dict(name="ldpc128_64_d64", kind="decode", code="ldpc128_64", d=64, layers=6, variant="aap", batch=10007),
        # the ECCT baseline's configuration of the model, an odd batch
        dict(name="polar64_32_ecct", kind="decode", code="polar64_32", d=64, layers=6, variant="ecct", batch=20011),
        # words that arrive in and leave to host memory
        dict(name="polar64_32_host", kind="host", code="polar64_32", d=64, layers=6, variant="aap", batch=30011),
        # all 60 weight tensors of the largest model quantised for export
        dict(name="ternarize_n10_d128", kind="ternarize", d=128, layers=10, weights=False),
        # the positional encoding of a newly drawn long code
        dict(name="spe_ldpc384_192", kind="spe", code="ldpc", n=384, d_spe=32),
    ]


def draw(rng):
    kind = rng.choices(("decode", "host", "ternarize", "spe"), (0.6, 0.12, 0.14, 0.14))[0]
    if kind == "ternarize":
        weights = rng.random() < 0.5
        d = rng.choice((32, 64, 128))
        return dict(kind=kind, d=d, layers=rng.randint(1, 5 if weights else 10), weights=weights)
    if kind == "spe":
        d_spe = rng.choice((8, 16, 32))
        code = rng.choice(("bch31_16", "polar64_32", "bch63_36", "ldpc", "ldpc"))
        if code != "ldpc":
            return dict(kind=kind, code=code, d_spe=d_spe)
        return dict(kind=kind, code=code, n=_log_even(rng, 48, 384), d_spe=d_spe)
    c = dict(kind=kind, code=rng.choice(("bch31_16", "polar64_32", "bch63_36", "ldpc", "ldpc")))
    if c["code"] == "ldpc":
        c["n"] = _log_even(rng, 48, 384)
    c["d"] = rng.choice((32, 64, 128))
    c["layers"] = rng.randint(2, 10)
    c["variant"] = rng.choices(("aap", "gelu", "fp", "ecct"), (0.55, 0.15, 0.15, 0.15))[0]
    # at most about a fifth of the largest listed case's arithmetic, less at the narrow widths
    # (whose time goes into attention rather than the contractions)
    word = _word_flops(dict(c, batch=1))
    top = min(60000, int(2e13 * (c["d"] / 128.0) ** 2 / word))
    c["batch"] = max(1, int(round(math.exp(rng.uniform(0.0, math.log(max(2, top)))))))
    return c


def _log_even(rng, lo, hi):
    return 2 * int(round(math.exp(rng.uniform(math.log(lo / 2), math.log(hi / 2)))))


# ------------------------------------------------------------------------------------------
# codes, models and inputs
# ------------------------------------------------------------------------------------------
_CODES, _MODELS = {}, {}

EBN0 = dict(bch31_16=4.0, polar64_32=4.0, bch63_36=4.0, ldpc128_64=3.0, ldpc384_192=2.5, ldpc=3.0)


def _code(case, seed=0):
    key = (case["code"], case.get("n"), seed)
    if key not in _CODES:
        if case["code"] == "ldpc":
            _CODES[key] = inputs.ldpc_regular_code(case["n"], case["n"] // 2, 3, 6, seed=case["n"] + 7919 * seed)
        else:
            _CODES[key] = inputs.make_code(case["code"])
    return _CODES[key]


def _model(case):
    """The deployed model of a decode case (fixed by the case; a user loads it once).  The long codes
    take a seeded table in the place of their positional encoding, whose host computation would
    take longer than everything else here."""
    key = tuple(case.get(k) for k in ("code", "n", "d", "layers", "variant"))
    if key not in _MODELS:
        code = _code(case)
        full = case["variant"] in ("fp", "ecct")
        m = inputs.random_model(code, case["d"], case["layers"], seed=1000 + case["d"] + case["layers"],
                                zero_frac=0.4 if case["code"] == "polar64_32" else 0.5,
                                activation=1 if case["variant"] in ("gelu", "ecct") else 0,
                                full_precision=full, spe_noise=code.T > 200)
        m.mask_mode = 1 if case["variant"] == "ecct" else 0
        _MODELS[key] = m
    return _MODELS[key]


def _received(case, seed):
    """Channel outputs of random codewords over BPSK and AWGN, on the GPU."""
    code = _code(case)
    g = torch.Generator(device="cuda").manual_seed(seed)
    G = torch.from_numpy(code.G).cuda().float()
    y = torch.empty((case["batch"], code.n), device="cuda")
    y.normal_(generator=g).mul_(inputs.awgn_sigma(EBN0[case["code"]], code.k / code.n))
    for s in range(0, case["batch"], 65536):
        part = y[s:s + 65536]
        msg = torch.randint(0, 2, (part.shape[0], G.shape[0]), device="cuda", generator=g).float()
        part += 1.0 - 2.0 * torch.remainder(msg @ G, 2.0)
    return y


def _shapes(case):
    d = case["d"]
    return [(d, d), (d, d), (d, d), (d, d), (4 * d, d), (d, 4 * d)] * case["layers"]


def _float_weights(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    w = [torch.randn(s, device="cuda", generator=g) / math.sqrt(s[1]) for s in _shapes(case)]
    delta = np.random.default_rng(seed).uniform(0.8, 2.2, len(w)).astype(np.float32)
    return w, delta


def _spe_inputs(case, seed):
    code = _code(case, seed % 1000 if case["code"] == "ldpc" else 0)  # a drawn code for each seed
    return code.H, inputs.spe_params(code.H, case["d_spe"], seed)


def prepare(case, seed):
    if case["kind"] == "ternarize":
        w, delta = _float_weights(case, seed)
        return dict(case=case, w=w, delta=delta)
    if case["kind"] == "spe":
        H, params = _spe_inputs(case, seed)
        return dict(case=case, H=H, params=params)
    y = _received(case, seed)
    return dict(case=case, dec=aecct.Decoder(_model(case)), y=y.cpu().numpy() if case["kind"] == "host" else y)


def run(state):
    kind = state["case"]["kind"]
    if kind == "decode":
        return state["dec"].decode(state["y"])  # bits, syndromes, logits
    if kind == "host":
        return state["dec"].decode_host(state["y"])
    if kind == "ternarize":  # codes, scales, and the forward weights where they are wanted
        return aecct.aap_ternarize(state["w"], state["delta"], 1e-8, want_weights=state["case"]["weights"])
    return aecct.spe_table(state["H"], state["params"])


# ------------------------------------------------------------------------------------------
# the work of a pass
# ------------------------------------------------------------------------------------------
def _masks(H, code_aware):
    """First-ring and second-ring masks [T, T] (Sec. 4.2), or the code-aware mask twice (Sec. 3)."""
    m, n = H.shape
    h = H.astype(np.int64)
    m1, m2 = np.zeros((n + m, n + m), bool), np.zeros((n + m, n + m), bool)
    m1[:n, n:], m1[n:, :n] = h.T > 0, h > 0
    m2[:n, :n], m2[n:, n:] = h.T @ h > 0, h @ h.T > 0
    return (m1 | m2, m1 | m2) if code_aware else (m1, m2)


def _word_flops(case):
    """Multiply-adds (counted as two) of one word: the linear layers, and the masked attention's
    dot products and weighted sums."""
    code = _code(case)
    m1, m2 = _masks(code.H, case["variant"] == "ecct")
    keys = (HEADS // 2) * (int(m1.sum()) + int(m2.sum()))
    return case["layers"] * (24.0 * code.T * case["d"] ** 2 + 4.0 * keys * (case["d"] // HEADS))


def work(case):
    if case["kind"] == "ternarize":
        size = sum(a * b for a, b in _shapes(case))
        return dict(bytes=size * (4.25 + (4.0 if case["weights"] else 0.0)), flops=2.0 * size)
    if case["kind"] == "spe":
        T = _code(case).T
        # the matrix in, the table out; a symmetric eigendecomposition with all vectors (about 9 T^3),
        # and for every node 4 heads of T x T scores, exponentials and weighted sums
        return dict(bytes=float(_code(case).H.size + 4 * T * case["d_spe"]), flops=9.0 * T ** 3 + 4.0 * T * T * T * 20.0)
    code, B = _code(case), case["batch"]
    weights = case["layers"] * 12 * case["d"] ** 2 * (2.0 if case["variant"] in ("fp", "ecct") else 0.25)
    return dict(bytes=weights + B * (4.0 * code.n + code.n + code.m + 4.0 * code.n), flops=B * _word_flops(case))


def tolerance(case):
    if case["kind"] == "ternarize":
        return "exact"  # order statistics, one product and one rounded quotient: nothing is summed
    if case["kind"] == "spe":
        return dict(rel=1.2e-7, max=1e-5)  # a table in 32 bits of a computation in 64
    if case["variant"] in ("fp", "ecct"):
        # 32-bit sums in another order, then activations rounded to bf16 in every layer
        return dict(rel=2.5e-2, max=0.5, differ=5e-3)
    # ternary linears: the ABI fixes one order of 32-bit operations, so that every implementation
    # of it gives the same bits (a quantised code that rounds the other way changes all that follows)
    return "exact"


# ------------------------------------------------------------------------------------------
# the same values in 64 bits
# ------------------------------------------------------------------------------------------
def exact(case, seed):
    if case["kind"] == "ternarize":
        return _exact_ternarize(case, seed)
    if case["kind"] == "spe":
        return _exact_spe(case, seed)
    code = _code(case)
    dense = case["layers"] * code.T * (24.0 * case["d"] ** 2 + 4.0 * code.T * case["d"])
    if case["batch"] * dense > 5e12:  # more than a few seconds in 64 bits
        return None
    return None, None, decode64(_model(case), _received(case, seed))


def decode64(model, y):
    """The decoder's logits in float64: dense masked attention, the quantiser (or the rounding of
    GEMM inputs to bf16) where the model has one."""
    dev = y.device
    f64 = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev, torch.float64)  # noqa: E731
    m, n = model.H.shape
    d, T = model.d, m + n
    dh = d // HEADS
    full = model.linear_mode == 1
    masks = torch.from_numpy(np.stack([_masks(model.H, model.mask_mode == 1)[e >= model.h_first]
                                       for e in range(HEADS)])).to(dev)
    H, emb, spe = f64(model.H), f64(model.emb), f64(model.spe)

    def weight(l, g):
        if full:
            return torch.from_numpy(model.w_full[l][g]).to(dev).bfloat16().double()
        return f64(model.w_tern[l][g])

    W = [[weight(l, g) for g in range(6)] for l in range(model.n_layers)]

    def operand(x):
        if full:
            return x.float().bfloat16().double(), 1.0
        a = x.abs().amax(-1, keepdim=True).clamp_min(float(np.float32(model.alpha_floor)))
        return torch.round(x * (127.0 / a)), a / 127.0

    def norm(v, g, b):
        v = v - v.mean(-1, keepdim=True)
        return v / torch.sqrt(v.square().mean(-1, keepdim=True) + float(np.float32(model.ln_eps))) * f64(g) + f64(b)

    out = torch.empty((y.shape[0], n), dtype=torch.float64, device=dev)
    step = max(1, int(1e9 / (8.0 * HEADS * T * T)))
    for s in range(0, y.shape[0], step):
        yb = y[s:s + step].double()
        synd = torch.remainder((yb < 0).double() @ H.T, 2.0)
        h = torch.cat([yb.abs(), 1.0 - 2.0 * synd], 1)
        x = torch.cat([h[..., None] * emb, spe.expand(yb.shape[0], -1, -1)], 2)
        for l in range(model.n_layers):
            def lin(q, f, g):
                v = q @ W[l][g].T
                return (v if full else v * (f * float(model.w_scale[l, g]))) + f64(model.bias[l][g])

            q, f = operand(x)
            Q, K, V = (lin(q, f, g).view(-1, T, HEADS, dh).transpose(1, 2) for g in range(3))
            S = (Q @ K.transpose(2, 3) / math.sqrt(dh)).masked_fill(~masks, -math.inf)
            A = (torch.softmax(S, -1) @ V).transpose(1, 2).reshape(-1, T, d)
            x = norm(x + lin(*operand(A), 3), model.ln_gamma[l, 0], model.ln_beta[l, 0])
            u = lin(*operand(x), 4)
            u = torch.relu(u) if model.activation == 0 else torch.nn.functional.gelu(u)
            x = norm(x + lin(*operand(u), 5), model.ln_gamma[l, 1], model.ln_beta[l, 1])
        out[s:s + step] = (x @ f64(model.w_d1) + model.b_d1) @ f64(model.w_out) + f64(model.b_out)
    return out


def _exact_ternarize(case, seed):
    w, delta = _float_weights(case, seed)
    scales, weights = [], []
    for t, dl in zip(w, delta):
        a = t.double().abs().reshape(-1).sort().values
        pos = 0.5 * (a.numel() - 1)
        lo = int(pos)
        gamma = a[lo] + (pos - lo) * (a[min(lo + 1, a.numel() - 1)] - a[lo])
        sc = gamma * float(dl)
        scales.append(sc)
        weights.append(torch.clamp(torch.round(t.double() / (sc + 1e-8)), -1.0, 1.0) * sc)
    return None, torch.stack(scales), weights if case["weights"] else None


def _exact_spe(case, seed):
    H, p = _spe_inputs(case, seed)
    m, n = H.shape
    T = n + m
    A = np.zeros((T, T))
    A[:n, n:], A[n:, :n] = H.T, H
    lam, U = np.linalg.eigh(np.diag(A.sum(1)) - A)
    # the canonical basis of each cluster of equal eigenvalues: Gram-Schmidt of its projector's
    # columns in node order
    tol, i = 1e-8 * max(1.0, float(np.abs(lam).max())), 0
    basis = np.zeros((T, T))
    while i < T:
        j = i + 1
        while j < T and lam[j] - lam[j - 1] <= tol:
            j += 1
        P, got = U[:, i:j] @ U[:, i:j].T, i
        for node in range(T):
            v, Q = P[:, node], basis[:, i:got]
            v = v - Q @ (Q.T @ v)
            v = v - Q @ (Q.T @ v)
            if np.linalg.norm(v) > 1e-6:
                basis[:, got] = v / np.linalg.norm(v)
                got += 1
                if got == j:
                    break
        i = j
    to = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    lam_t, U_t, w_pe = to(lam), to(basis), to(p.w_pe)
    out = torch.empty((T, w_pe.shape[1]), dtype=torch.float64, device="cuda")
    for node in range(T):
        X = torch.stack([lam_t, U_t[node]], 1) @ w_pe
        Q, K, V = (X @ to(w) for w in (p.wq, p.wk, p.wv))  # [heads, T, d_e]
        S = torch.softmax(Q @ K.transpose(1, 2) / math.sqrt(Q.shape[2]), -1)
        out[node] = (S @ V).mean(1).reshape(-1) @ to(p.wo)
    return out
