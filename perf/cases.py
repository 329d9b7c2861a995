"""Timed cases of the decoder: what its users run, from one syndrome to a million.

A case names a decoding problem of `workloads`, the call made on it and the
size of the batch.  The calls are the public ones: `BeamSearchDecoder.decode`
(device tensors), `decode_host_ptrs` (pinned host buffers, copies inside),
`bp_llr` (plain BP) and `unrolled_loss` with its backward (training).
"""
import functools
import math

import numpy as np
import torch

from paper_2512_07057_gb300 import binding, decoder, unrolled, workloads

ALPHA = 0.625

# Mean BP iterations of the sequential algorithm per shot at a few noise rates
# (code, preset family): the work a decode cannot do without.
MEAN_ITERS = {
    "bb72": [(0.03, 4.5)],
    "bb144": [(0.01, 1.15), (0.03, 4.86), (0.05, 47.9)],
    "phenom": [(0.001, 1.06), (0.002, 1.23), (0.003, 1.47)],
    "synthetic": [(0.0, 1.15)],
    "xyz": [(0.03, 20.3), (0.05, 23.9)],
    "bb144_many": [(0.03, 13580.0), (0.05, 13460.0)],
}
PRECISION = {"fp32": binding.BSD_FP32, "fp16": binding.BSD_FP16, "bf16": binding.BSD_BF16}


def _case(call, code, p, preset, shots, **more):
    c = {"call": call, "code": code, "p": p, "preset": preset, "shots": shots, "precision": "fp32", "iters": 0, "ckpt": 0}
    c.update(more)
    return c


def listed():
    def named(name, c):
        return {"name": name, **c}

    return [
        # one syndrome at a time: a decoder in the loop of an experiment, latency bound
        named("bb144_one", _case("decode", "bb144", 0.03, "beam32_340iters", 1)),
        # a handful of circuit-shaped syndromes: a control system that collects a few shots per call
        named("synthetic_few", _case("decode", "synthetic", 0.0, "beam64_640iters", 37)),
        # the small code of a first study, 10^4 shots
        named("bb72_10k", _case("decode", "bb72", 0.03, "bb72", 10_000)),
        # the large code-capacity sweep at its hardest noise rate: most of the time is beam rounds
        named("bb144_1m", _case("decode", "bb144", 0.05, "beam32_340iters", 1_000_000)),
        # the same sweep fed from pinned host memory at a middle noise rate, a ragged batch
        named("bb144_host", _case("host", "bb144", 0.03, "beam32_340iters", 300_007)),
        # repeated syndrome measurement, widest single-result preset, single precision
        named("phenom_100k", _case("decode", "phenom", 0.003, "beam64_640iters", 100_000)),
        # the same with half-precision messages and near-tie re-runs, a ragged batch
        named("phenom_fp16", _case("decode", "phenom", 0.002, "beam64_640iters", 49_999, precision="fp16")),
        # a circuit-shaped detector error model, 10^6 shots: logical error rate estimation
        named("synthetic_1m", _case("decode", "synthetic", 0.0, "beam32_340iters", 1_000_000)),
        # both error types of depolarizing noise decoded together
        named("xyz_100k", _case("decode", "xyz", 0.05, "beam64_640iters", 100_000)),
        # 32 solutions per shot: every shot stays in the beam for all rounds
        named("bb144_32results", _case("decode", "bb144", 0.03, "beam64_32res_640iters", 3_001)),
        # posteriors of plain BP after a fixed number of iterations
        named("llr_phenom", _case("llr", "phenom", 0.002, "beam64_640iters", 8_191, iters=20)),
        # one training step of the unrolled decoder: forward, loss terms, weight gradients
        named("train_phenom", _case("train", "phenom", 0.002, "", 4_096, iters=20, ckpt=5)),
    ]


def _size(rng, lo, hi):
    """A size spread over the logarithm of [lo, hi]; every other one odd."""
    n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    return max(lo, min(hi, n | 1 if rng.random() < 0.5 else n))


def draw(rng):
    kind = rng.choice(["few", "bb72", "bb144", "host", "phenom", "phenom16", "synthetic", "xyz", "many", "llr", "train"])
    preset = rng.choice(["beam8_230iters", "beam32_340iters", "beam64_640iters"])
    if kind == "few":
        code = rng.choice(["bb144", "phenom", "synthetic", "xyz"])
        p = {"bb144": rng.uniform(0.01, 0.05), "phenom": rng.uniform(0.001, 0.003), "synthetic": 0.0,
             "xyz": rng.uniform(0.03, 0.05)}[code]
        return _case("decode", code, round(p, 5), preset, _size(rng, 1, 64))
    if kind == "bb72":
        return _case("decode", "bb72", 0.03, "bb72", _size(rng, 500, 20_000))
    if kind == "bb144":
        return _case("decode", "bb144", round(rng.uniform(0.01, 0.05), 4), preset, _size(rng, 1_000, 600_000))
    if kind == "host":
        return _case("host", "bb144", round(rng.uniform(0.01, 0.05), 4), "beam32_340iters", _size(rng, 1_000, 300_000))
    if kind == "phenom":
        return _case("decode", "phenom", round(rng.uniform(0.001, 0.003), 5), preset, _size(rng, 1_000, 100_000))
    if kind == "phenom16":
        return _case("decode", "phenom", round(rng.uniform(0.001, 0.003), 5), preset, _size(rng, 1_000, 100_000),
                     precision=rng.choice(["fp16", "bf16"]))
    if kind == "synthetic":
        return _case("decode", "synthetic", 0.0, preset, _size(rng, 1_000, 1_000_000))
    if kind == "xyz":
        return _case("decode", "xyz", round(rng.uniform(0.03, 0.05), 4), "beam64_640iters", _size(rng, 1_000, 100_000))
    if kind == "many":
        return _case("decode", "bb144", round(rng.uniform(0.03, 0.05), 4), "beam64_32res_640iters", _size(rng, 200, 3_000))
    if kind == "llr":
        code = rng.choice(["bb144", "phenom"])
        p = rng.uniform(0.01, 0.05) if code == "bb144" else rng.uniform(0.001, 0.003)
        return _case("llr", code, round(p, 5), preset, _size(rng, 200, 8_000), iters=rng.randint(5, 20))
    iters = rng.randint(8, 20)
    return _case("train", "phenom", round(rng.uniform(0.001, 0.003), 5), "", _size(rng, 256, 4_096), iters=iters,
                 ckpt=rng.randint(2, 6))


@functools.lru_cache(maxsize=16)
def _problem(code, p):
    if code == "bb72":
        return workloads.bb72_code_capacity(p)
    if code == "bb144":
        return workloads.bb144_code_capacity(p)
    if code == "phenom":
        return workloads.bb_phenomenological(12, 6, 12, p, p)
    if code == "synthetic":
        return workloads.synthetic_dem()
    return workloads.bb_xyz_code_capacity(12, 6, p)


def _pack(bits):
    """0/1 tensor [B, L] -> int32 words [B, ceil(L/32)], bit i in word i // 32."""
    nb, length = bits.shape
    width = (length + 31) // 32
    b = torch.zeros((nb, width * 32), dtype=torch.int64, device=bits.device)
    b[:, :length] = bits
    w = (b.view(nb, width, 32) << torch.arange(32, device=bits.device)).sum(-1)
    return torch.where(w >= 2 ** 31, w - 2 ** 32, w).to(torch.int32)


def _shots(prob, nshots, seed, keep_errors=False):
    """Syndromes (and errors) of nshots shots, e_j ~ Bernoulli(p_j), as CUDA bit words."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    ht = torch.from_numpy(prob.H_dense()).cuda().t().to(torch.float16).contiguous()
    p = torch.from_numpy(prob.priors).cuda().float()
    synd = torch.empty((nshots, (prob.M + 31) // 32), dtype=torch.int32, device="cuda")
    errs = torch.empty((nshots, (prob.N + 31) // 32), dtype=torch.int32, device="cuda") if keep_errors else None
    step = max(1, (1 << 27) // prob.N)
    for a in range(0, nshots, step):
        n = min(step, nshots - a)
        e = torch.rand((n, prob.N), generator=g, device="cuda") < p
        s = e.to(torch.float16) @ ht          # counts below 2048: exact
        synd[a:a + n] = _pack(s.to(torch.int64) & 1)
        if keep_errors:
            errs[a:a + n] = _pack(e)
    return synd, errs


def _weights(prob, case, seed):
    """Weights some steps into training: the scale with a few per cent of spread."""
    g = torch.Generator(device="cuda").manual_seed(seed + 1)
    return ALPHA * (1 + 0.05 * torch.randn((case["iters"], prob.n_edges), generator=g, device="cuda"))


def prepare(case, seed):
    prob = _problem(case["code"], case["p"])
    if case["call"] == "train":
        synd, errs = _shots(prob, case["shots"], seed, keep_errors=True)
        return {"call": "train", "synd": synd, "errs": errs, "w": _weights(prob, case, seed).requires_grad_(True),
                "trainer": unrolled.UnrolledTrainer(prob, case["shots"], T=case["iters"], ckpt_every=case["ckpt"])}
    if case["preset"] == "bb72":
        params = decoder.make_params(max_rounds=10, beam_width=8, initial_iters=50, iters_per_round=20, ms_scale=ALPHA)
    else:
        params = decoder.make_params(case["preset"], ms_scale=ALPHA, msg_precision=PRECISION[case["precision"]])
    state = {"call": case["call"], "dec": decoder.BeamSearchDecoder(prob, params)}
    state["synd"], _ = _shots(prob, case["shots"], seed)
    if case["call"] == "llr":
        state["iters"] = case["iters"]
    if case["call"] == "host":
        def pinned(*shape):
            return torch.empty(shape, dtype=torch.int32, pin_memory=True)

        nb = case["shots"]
        host = pinned(*state["synd"].shape)
        host.copy_(state["synd"])
        state.update(synd=host, corr=pinned(nb, (prob.N + 31) // 32), obs=pinned(nb, (prob.K + 31) // 32),
                     status=pinned(nb), its=pinned(nb))
    return state


def run(state):
    if state["call"] == "train":
        w = state["w"]
        w.grad = None
        losses = unrolled.unrolled_loss(w, state["trainer"], state["synd"], state["errs"])
        losses[0].backward()
        return {"loss": losses.detach(), "grad": w.grad}
    dec = state["dec"]
    if state["call"] == "llr":
        llr, total = dec.bp_llr(state["synd"], state["iters"])
        return {"llr": llr, "sum": total}
    if state["call"] == "host":
        s = state["synd"]
        dec.decode_host_ptrs(s.data_ptr(), s.shape[0], state["corr"].data_ptr(), state["obs"].data_ptr(),
                             state["status"].data_ptr(), state["its"].data_ptr())
        return {"corrections": state["corr"], "obs": state["obs"], "status": state["status"], "iters": state["its"]}
    out = dec.decode(state["synd"])
    return {"corrections": out.corrections, "obs": out.obs_flips, "status": out.status, "iters": out.iters}


def _mean_iters(case):
    key = "bb144_many" if "32res" in case["preset"] else case["code"]
    ps, its = zip(*MEAN_ITERS[key])
    return float(np.exp(np.interp(case["p"], ps, np.log(its))))


def work(case):
    """Bytes: every input and output once.  Operations: 6 per message update
    (two smallest magnitudes and the sign on the check side, two sums on the
    error side), 12 more per update for the adjoint of a training step."""
    prob = _problem(case["code"], case["p"])
    nb, edges = case["shots"], prob.n_edges
    wm, wn, wk = ((x + 31) // 32 for x in (prob.M, prob.N, prob.K))
    if case["call"] == "train":
        return {"bytes": 4 * (nb * (wm + wn) + 2 * case["iters"] * edges), "flops": 18.0 * nb * case["iters"] * edges}
    if case["call"] == "llr":
        return {"bytes": 4 * nb * (wm + 2 * prob.N), "flops": 6.0 * nb * case["iters"] * edges}
    return {"bytes": 4 * nb * (wm + wn + wk + 2), "flops": 6.0 * nb * edges * _mean_iters(case)}


class _Graph:
    """Padded neighbour tables of H on the GPU, edges in CSR order."""

    def __init__(self, prob):
        rows = np.repeat(np.arange(prob.M), np.diff(prob.H_row_ptr))
        cols = np.asarray(prob.H_col_idx)
        self.E = len(cols)
        self.row = torch.from_numpy(rows).cuda()
        self.col = torch.from_numpy(cols.astype(np.int64)).cuda()
        by_row = np.full((prob.M, int(np.diff(prob.H_row_ptr).max())), self.E, np.int64)
        by_row[rows, np.arange(self.E) - np.asarray(prob.H_row_ptr)[rows]] = np.arange(self.E)
        self.by_row = torch.from_numpy(by_row).cuda()
        self.at = torch.from_numpy(np.arange(self.E) - np.asarray(prob.H_row_ptr)[rows]).cuda()
        order = np.argsort(cols, kind="stable")
        start = np.searchsorted(cols[order], np.arange(prob.N))
        by_col = np.full((prob.N, int(np.bincount(cols, minlength=prob.N).max())), self.E, np.int64)
        by_col[cols[order], np.arange(self.E) - start[cols[order]]] = order
        self.by_col = torch.from_numpy(by_col).cuda()
        p = torch.from_numpy(np.asarray(prob.priors)).cuda()
        self.lam = torch.log((1 - p) / p)

    def check(self, msg, flip):
        """(-1)^s_i times the product of the other signs times the smallest other magnitude; [B, E] in and out."""
        limit = 1e4
        pad = torch.cat([msg, torch.full_like(msg[:, :1], math.inf)], 1)[:, self.by_row]     # [B, M, D]
        mag, neg = pad.abs(), (pad < 0)
        low = mag.amin(-1, keepdim=True)
        first = (mag == low).to(torch.uint8).argmax(-1, keepdim=True)
        low = torch.gather(mag, -1, first)
        rest = mag.scatter(-1, first, math.inf)
        best = rest.amin(-1, keepdim=True)
        low2 = torch.gather(mag, -1, (rest == best).to(torch.uint8).argmax(-1, keepdim=True))
        low2 = torch.where(torch.isinf(best), torch.full_like(low2, limit), low2)     # no other neighbour
        here = self.at[None, :] == first[:, self.row, 0]
        value = torch.where(here, low2[:, self.row, 0], low[:, self.row, 0])
        odd = (neg.sum(-1)[:, self.row] + (msg < 0) + flip[:, self.row]) & 1
        return value * (1 - 2 * odd).to(value.dtype)

    def update(self, d):
        """(E, Lambda) of Eqs. 2-3 from the check messages [B, E]."""
        total = self.lam + torch.cat([d, torch.zeros_like(d[:, :1])], 1)[:, self.by_col].sum(-1)
        return (total[:, self.col] - d).clamp(-1e4, 1e4), total


def _bits(words, length):
    w = words.to(torch.int64) & 0xFFFFFFFF
    b = (w[:, :, None] >> torch.arange(32, device=w.device)) & 1
    return b.reshape(w.shape[0], -1)[:, :length]


def exact(case, seed):
    if case["call"] not in ("llr", "train"):
        return None
    prob = _problem(case["code"], case["p"])
    g = _Graph(prob)
    nb, iters = case["shots"], case["iters"]
    synd, errs = _shots(prob, nb, seed, keep_errors=True)
    flips = _bits(synd, prob.M)
    if case["call"] == "llr":
        llr, total = [], []
        for a in range(0, nb, 1024):
            flip = flips[a:a + 1024]
            msg = g.lam[g.col].expand(flip.shape[0], -1)
            acc = 0
            for _ in range(iters):
                msg, post = g.update(ALPHA * g.check(msg, flip))
                acc = acc + post
            llr.append(post)
            total.append(acc)
        return {"llr": torch.cat(llr), "sum": torch.cat(total)}
    w = _weights(prob, case, seed).double().requires_grad_(True)
    terms = torch.zeros(iters, dtype=torch.float64, device="cuda")
    for a in range(0, nb, 256):
        flip, err = flips[a:a + 256], _bits(errs[a:a + 256], prob.N).double()
        msg = g.lam[g.col].expand(flip.shape[0], -1)
        loss = []
        for t in range(iters):
            msg, post = g.update(w[t] * g.check(msg, flip))
            loss.append(torch.nn.functional.binary_cross_entropy_with_logits(-post, err, reduction="sum") / (nb * prob.N))
        loss = torch.stack(loss)
        loss.sum().backward()
        terms += loss.detach()
    return {"loss": torch.cat([terms.sum()[None], terms]), "grad": w.grad}
