"""The measured work of this framework: what a user has it do, through its public entry points.

Every case is one call (or the short call sequence of one homomorphic operation) on data that is
already in device memory, as the ciphertexts of a running program are.  A program creates its
context, parameter sets, conversion plans and the HE-Mult workspaces once and uses them for all
its data, so these are made at the first state that needs them and shared by the later ones;
inputs, keys, outputs and the plans that name buffers belong to one state.
"""
from __future__ import annotations

import functools

import numpy as np
import torch

from paper_2501_07047_gb300 import hefx, inputs
from paper_2501_07047_gb300.hemult import HeMult, digit_ranges

SERVE_SPECIAL = 8   # special primes of a serving request
SERVE_LMAX = 36     # ciphertext limbs of the largest serving request
BATCH_LMAX = 32     # limbs of the largest job of an uneven batch


def listed():
    return [
        # one product of two polynomials of the smallest ring in use, one limb: the latency of a call
        {"name": "polymul_n12_l1_b1", "op": "polymul", "logn": 12, "bits": 28, "limbs": 1, "batch": 1},
        # the paper's Set B and Set C transforms (8 limbs of 2^13, 15 limbs of 2^14, 16 polynomials):
        # ciphertexts of shallow circuits, a row per CTA and a row per small cluster
        {"name": "ntt_fwd_n13_l8_b16", "op": "ntt_fwd", "logn": 13, "bits": 28, "limbs": 8, "batch": 16},
        {"name": "ntt_inv_n14_l15_b16", "op": "ntt_inv", "logn": 14, "bits": 28, "limbs": 15, "batch": 16},
        # one polynomial of the bootstrappable ring: what a single ciphertext operation transforms
        {"name": "ntt_fwd_n16_l24_b1", "op": "ntt_fwd", "logn": 16, "bits": 28, "limbs": 24, "batch": 1},
        # the benchmark's batch of 8 such polynomials, both directions
        {"name": "ntt_fwd_n16_l24_b8", "op": "ntt_fwd", "logn": 16, "bits": 28, "limbs": 24, "batch": 8},
        {"name": "ntt_inv_n16_l24_b8", "op": "ntt_inv", "logn": 16, "bits": 28, "limbs": 24, "batch": 8},
        # the largest ring, with 30-bit moduli: products of a batch of polynomials
        {"name": "polymul_n17_l24_b4", "op": "polymul", "logn": 17, "bits": 30, "limbs": 24, "batch": 4},
        # RNS basis conversion of a batch to the special primes, and the paper's widest conversion
        {"name": "bconv_24to8_b16", "op": "bconv", "logn": 16, "src": 24, "dst": 8, "batch": 16},
        {"name": "bconv_24to56_b8", "op": "bconv", "logn": 16, "src": 24, "dst": 56, "batch": 8},
        # 256 independent products of uneven ring degrees (2^12 .. 2^16) and limb counts (4 .. 32)
        {"name": "batch_256_jobs", "op": "batch", "jobs": 256, "shapes": 4},
        # HE-Mult with key switching and Rescale at the paper's (L, log q, dnum) = (48, 28, 3)
        {"name": "hemult_n16_l48_k16", "op": "hemult", "logn": 16, "limbs": 48, "alpha": 16},
        # a serving group: the front halves of 8 requests of uneven limb counts in shared launches
        {"name": "serve_n15_r8", "op": "serve", "logn": 15, "requests": 8, "shapes": 5},
    ]


def draw(rng):
    def log_between(lo, hi):
        return int(round(lo * (hi / lo) ** rng.random()))

    op = rng.choice(["ntt_fwd", "ntt_inv", "ntt_fwd", "ntt_inv", "polymul", "polymul", "bconv", "bconv", "batch",
                     "hemult", "serve"])
    if op in ("ntt_fwd", "ntt_inv", "polymul"):
        logn = rng.randint(12, 17)
        limbs = log_between(1, 48)
        room = (1 << 25) // (limbs << logn)  # residues of one operand
        return {"op": op, "logn": logn, "bits": rng.choice([28, 28, 28, 30]), "limbs": limbs,
                "batch": log_between(1, max(1, min(32, room)))}
    if op == "bconv":
        src, dst = rng.randint(4, 24), rng.randint(4, 56)
        logn = rng.randint(13, 16)
        room = (1 << 25) // ((src + dst) << logn)
        return {"op": op, "logn": logn, "src": src, "dst": dst, "batch": log_between(1, max(1, min(16, room)))}
    if op == "batch":
        return {"op": op, "jobs": log_between(8, 224), "shapes": rng.randint(100, 10 ** 6)}
    if op == "hemult":
        limbs = rng.randint(6, 48)
        return {"op": op, "logn": rng.randint(14, 16), "limbs": limbs, "alpha": -(-limbs // rng.choice([3, 4]))}
    return {"op": op, "logn": rng.randint(13, 16), "requests": log_between(1, 16), "shapes": rng.randint(100, 10 ** 6)}


# ----------------------------------------------------------------------------- what a program keeps

@functools.lru_cache(maxsize=None)
def _ctx():
    return hefx.hefx_create(0)


@functools.lru_cache(maxsize=None)
def _primes(count, bits, logn):
    return tuple(inputs.ntt_primes(count, bits, 1 << 17 if logn <= 16 else 2 << logn))


@functools.lru_cache(maxsize=None)
def _params(logn, primes):
    return hefx.hefx_params_create(_ctx(), logn, primes)


@functools.lru_cache(maxsize=None)
def _bconv_plan(logn, src, dst):
    return hefx.hefx_bconv_plan_create(_ctx(), logn, src, dst)


@functools.lru_cache(maxsize=None)
def _hemult(logn, limbs, alpha):
    return HeMult(_ctx(), logn, _primes(limbs, 28, logn), _primes(alpha, 30, logn), alpha)


@functools.lru_cache(maxsize=None)
def _serve_slots():
    return hefx.hefx_mult_batch_create(_ctx(), 32, SERVE_LMAX)


# ----------------------------------------------------------------------------- inputs

def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _residues(gen, batch, primes, n):
    """[batch][limb][n], limb i uniform in [0, primes[i]): the residues of a ciphertext."""
    q = torch.tensor(primes, dtype=torch.int64, device="cuda")[None, :, None]
    return (torch.randint(0, 1 << 62, (batch, len(primes), n), generator=gen, device="cuda") % q).to(torch.int32)


def _empty(*shape):
    return torch.empty(shape, dtype=torch.int32, device="cuda")


def _batch_shapes(case):
    return inputs.uneven_jobs(case["shapes"], case["jobs"], lmin=4, lmax=BATCH_LMAX)


def _serve_limbs(case):
    r = inputs.splitmix64(case["shapes"], case["requests"])
    return [8 + int(v % np.uint64(SERVE_LMAX - 8 + 1)) for v in r]


class State:
    """Buffers and handles of one state; `plan`, where there is one, names its buffers."""

    plan = destroy = None

    def __del__(self):
        if self.plan is not None:
            self.destroy(self.plan)
            self.plan = None


def _in_ntt(case, seed):
    primes = _primes(case["limbs"], case["bits"], case["logn"])
    return _residues(_generator(seed), case["batch"], primes, 1 << case["logn"]), primes


def _in_polymul(case, seed):
    primes, n = _primes(case["limbs"], case["bits"], case["logn"]), 1 << case["logn"]
    gen = _generator(seed)
    return _residues(gen, case["batch"], primes, n), _residues(gen, case["batch"], primes, n), primes


def _in_bconv(case, seed):
    src, dst = _primes(case["src"], 28, case["logn"]), _primes(case["dst"], 30, case["logn"])
    return _residues(_generator(seed), case["batch"], src, 1 << case["logn"]), src, dst


def _in_batch(case, seed):
    gen, primes = _generator(seed), _primes(BATCH_LMAX, 28, 16)
    return [(logn, L, _residues(gen, 1, primes[:L], 1 << logn)[0], _residues(gen, 1, primes[:L], 1 << logn)[0])
            for logn, L in _batch_shapes(case)], primes


def _in_hemult(case, seed):
    gen, n = _generator(seed), 1 << case["logn"]
    qs, ps = _primes(case["limbs"], 28, case["logn"]), _primes(case["alpha"], 30, case["logn"])
    dnum = len(digit_ranges(len(qs), case["alpha"]))
    cts = [_residues(gen, 1, qs, n)[0] for _ in range(4)]
    evk = _residues(gen, 2 * dnum, qs + ps, n).reshape(dnum, 2, len(qs) + len(ps), n)
    return cts, evk, qs, ps


def _in_serve(case, seed):
    gen, n = _generator(seed), 1 << case["logn"]
    qall, ps = _primes(SERVE_LMAX, 28, case["logn"]), _primes(SERVE_SPECIAL, 30, case["logn"])
    key_q = [_residues(gen, 1, qall, n)[0] for _ in range(2)]
    key_p = [_residues(gen, 1, ps, n)[0] for _ in range(2)]
    cts = [[_residues(gen, 1, qall[:L], n)[0] for _ in range(4)] for L in _serve_limbs(case)]
    return cts, key_q, key_p, qall, ps


# ----------------------------------------------------------------------------- the measured calls

def prepare(case, seed):
    s, ctx, op = State(), _ctx(), case["op"]
    s.op, s.ctx = op, ctx
    if op in ("ntt_fwd", "ntt_inv"):
        s.data, primes = _in_ntt(case, seed)
        s.params, s.batch = _params(case["logn"], primes), case["batch"]
    elif op == "polymul":
        s.a, s.b, primes = _in_polymul(case, seed)
        s.c = torch.empty_like(s.a)
        s.params, s.batch = _params(case["logn"], primes), case["batch"]
    elif op == "bconv":
        s.x, src, dst = _in_bconv(case, seed)
        s.y = _empty(case["batch"], len(dst), 1 << case["logn"])
        s.conv, s.batch = _bconv_plan(case["logn"], src, dst), case["batch"]
    elif op == "batch":
        s.jobs, primes = _in_batch(case, seed)
        s.out = _empty(sum(L << logn for logn, L, _, _ in s.jobs))  # the jobs' products, one after another
        parts = s.out.split([L << logn for logn, L, _, _ in s.jobs])
        s.plan = hefx.hefx_batch_plan_create(
            ctx, [(_params(logn, primes), L, a, b, c) for (logn, L, a, b), c in zip(s.jobs, parts)])
        s.destroy = hefx.hefx_batch_plan_destroy
        s.stream = torch.cuda.Stream()  # the plan replays its graph on a stream of the program's own
    elif op == "hemult":
        s.cts, s.evk, qs, _ = _in_hemult(case, seed)
        s.hm = _hemult(case["logn"], case["limbs"], case["alpha"])
        s.out = _empty(2, len(qs) - 1, 1 << case["logn"])
    elif op == "serve":
        s.cts, s.key_q, s.key_p, qall, ps = _in_serve(case, seed)
        n, logn = 1 << case["logn"], case["logn"]
        limbs = _serve_limbs(case)
        s.plan = [hefx.hefx_mult_plan_create(ctx, _params(logn, qall[:L]), _params(logn, ps),
                                             _bconv_plan(logn, qall[:L], ps), s.key_q[0][:L], s.key_q[1][:L],
                                             s.key_p[0], s.key_p[1]) for L in limbs]
        s.destroy = lambda plans: [hefx.hefx_mult_plan_destroy(p) for p in plans]
        s.out = [_empty(4 * L + 2 * SERVE_SPECIAL, n) for L in limbs]
        s.work = [_empty(2 * L + SERVE_SPECIAL, n) for L in limbs]
        s.operands = [[c[i] for c in s.cts] for i in range(4)]
        s.slots = _serve_slots()
    else:
        raise ValueError(op)
    return s


def run(s):
    st = torch.cuda.current_stream()
    if s.op == "ntt_fwd":
        hefx.hefx_ntt_fwd(s.ctx, s.params, s.data, s.batch, stream=st)  # in place
        return s.data
    if s.op == "ntt_inv":
        hefx.hefx_ntt_inv(s.ctx, s.params, s.data, s.batch, stream=st)
        return s.data
    if s.op == "polymul":
        hefx.hefx_poly_mul(s.ctx, s.params, s.a, s.b, s.c, s.batch, stream=st)
        return s.c
    if s.op == "bconv":
        hefx.hefx_basis_convert(s.ctx, s.conv, s.x, s.y, s.batch, stream=st)
        return s.y
    if s.op == "batch":
        s.stream.wait_stream(st)
        hefx.hefx_batch_polymul(s.ctx, s.plan, s.stream)
        st.wait_stream(s.stream)
        return s.out
    if s.op == "hemult":
        s.hm.run(*s.cts, s.evk, s.out, st)
        return s.out
    hefx.hefx_mult_front_batch(s.ctx, s.slots, s.plan, *s.operands, s.out, s.work, st)
    return s.out


def work(case):
    """Each input (operands, keys) read once and each output written once, 4 bytes a residue.  The
    arithmetic is whole-number arithmetic, so no floating-point operation is needed."""
    op = case["op"]
    if op in ("ntt_fwd", "ntt_inv", "polymul"):
        words = (3 if op == "polymul" else 2) * case["batch"] * case["limbs"] << case["logn"]
    elif op == "bconv":
        words = case["batch"] * (case["src"] + case["dst"]) << case["logn"]
    elif op == "batch":
        words = 3 * sum(L << logn for logn, L in _batch_shapes(case))
    elif op == "hemult":
        L, K = case["limbs"], case["alpha"]
        words = (4 * L + 2 * len(digit_ranges(L, K)) * (L + K) + 2 * (L - 1)) << case["logn"]
    else:
        limbs = _serve_limbs(case)
        # four operands and the keys (shared by the requests) in; d0, d1 and the key products out
        words = (sum(8 * L + 2 * SERVE_SPECIAL for L in limbs) + 2 * max(limbs) + 2 * SERVE_SPECIAL) << case["logn"]
    return {"bytes": 4 * words, "flops": 0}


# ----------------------------------------------------------------------------- the same in 64-bit integers

def _root_2n(q, n):
    """psi = g^((q-1)/2N), g the smallest generator of Z_q^*."""
    rest, factors, d = q - 1, [], 2
    while d * d <= rest:
        if rest % d == 0:
            factors.append(d)
            while rest % d == 0:
                rest //= d
        d += 1
    factors += [rest] if rest > 1 else []
    g = next(g for g in range(2, q) if all(pow(g, (q - 1) // f, q) != 1 for f in factors))
    return pow(g, (q - 1) // (2 * n), q)


@functools.lru_cache(maxsize=4)
def _tables64(primes, n):
    """psi^brv(k) and psi^-brv(k), [limb][N]."""
    q = torch.tensor(primes, dtype=torch.int64, device="cuda")[:, None]
    k = torch.arange(n, device="cuda")
    rev = torch.zeros_like(k)
    for b in range(n.bit_length() - 1):
        rev |= ((k >> b) & 1) << (n.bit_length() - 2 - b)
    psi = [_root_2n(int(p), n) for p in primes]
    out = []
    for roots in (psi, [pow(r, -1, p) for r, p in zip(psi, primes)]):
        pw = torch.ones((len(primes), 1), dtype=torch.int64, device="cuda")
        while pw.shape[1] < n:
            step = torch.tensor([pow(r, pw.shape[1], p) for r, p in zip(roots, primes)], device="cuda")[:, None]
            pw = torch.cat([pw, pw * step % q], 1)
        out.append(pw[:, rev])
    return out


def _ntt64(x, primes):
    """Forward negacyclic NTT of x [..., limb, N] (int64): natural order in, bit-reversed out."""
    shape, L, n = x.shape, len(primes), x.shape[-1]
    q = torch.tensor(primes, dtype=torch.int64, device="cuda")[:, None, None]
    w = _tables64(tuple(primes), n)[0]
    x, m = x.reshape(-1, L, n), 1
    while m < n:
        v = x.reshape(-1, L, m, 2, n // (2 * m))
        t = v[..., 1, :] * w[:, m:2 * m, None] % q
        a = v[..., 0, :]
        x, m = torch.stack([(a + t) % q, (a - t + q) % q], -2), 2 * m
    return x.reshape(shape)


def _intt64(x, primes):
    shape, L, n = x.shape, len(primes), x.shape[-1]
    q = torch.tensor(primes, dtype=torch.int64, device="cuda")[:, None, None]
    w = _tables64(tuple(primes), n)[1]
    x, m = x.reshape(-1, L, n), n // 2
    while m >= 1:
        v = x.reshape(-1, L, m, 2, n // (2 * m))
        a, b = v[..., 0, :], v[..., 1, :]
        x, m = torch.stack([(a + b) % q, (a - b + q) * w[:, m:2 * m, None] % q], -2), m // 2
    ninv = torch.tensor([pow(n, -1, p) for p in primes], device="cuda")[:, None]
    return (x.reshape(-1, L, n) * ninv % q[..., 0]).reshape(shape)


def _bconv64(x, src, dst):
    """sum_i [x_i (Q/q_i)^-1]_{q_i} [Q/q_i]_{p_j} mod p_j, x [..., len(src), N]."""
    Q = 1
    for q in src:
        Q *= q
    hat = [Q // q for q in src]
    y = x * torch.tensor([pow(h % q, -1, q) for h, q in zip(hat, src)], device="cuda")[:, None]
    y = y % torch.tensor(src, dtype=torch.int64, device="cuda")[:, None]
    out = torch.empty((*x.shape[:-2], len(dst), x.shape[-1]), dtype=torch.int64, device="cuda")
    for j, p in enumerate(dst):
        acc = torch.zeros_like(out[..., j, :])
        for i, h in enumerate(hat):
            acc = (acc + y[..., i, :] * (h % p)) % p
        out[..., j, :] = acc
    return out


def _q64(primes):
    return torch.tensor(primes, dtype=torch.int64, device="cuda")[:, None]


def exact(case, seed):
    op = case["op"]
    if op in ("ntt_fwd", "ntt_inv"):
        x, primes = _in_ntt(case, seed)
        return (_ntt64 if op == "ntt_fwd" else _intt64)(x.long(), primes)
    if op == "polymul":
        a, b, primes = _in_polymul(case, seed)
        return _intt64(_ntt64(a.long(), primes) * _ntt64(b.long(), primes) % _q64(primes), primes)
    if op == "bconv":
        x, src, dst = _in_bconv(case, seed)
        return _bconv64(x.long(), src, dst)
    if op == "batch":
        jobs, primes = _in_batch(case, seed)
        out = []
        for logn, L, a, b in sorted(jobs, key=lambda j: j[0]):  # one table per ring degree at a time
            fa, fb = (torch.zeros((len(primes), 1 << logn), dtype=torch.int64, device="cuda") for _ in range(2))
            fa[:L], fb[:L] = a.long(), b.long()
            c = _intt64(_ntt64(fa, primes) * _ntt64(fb, primes) % _q64(primes), primes)
            out.append(c[:L].reshape(-1))
        order = sorted(range(len(jobs)), key=lambda j: jobs[j][0])
        return torch.cat([out[order.index(j)] for j in range(len(jobs))])
    if op == "hemult":
        (a0, a1, b0, b1), evk, qs, ps = _in_hemult(case, seed)
        a0, a1, b0, b1, evk = (t.long() for t in (a0, a1, b0, b1, evk))
        q, qp, L = _q64(qs), qs + ps, len(qs)
        d = torch.stack([a0 * b0 % q, (a0 * b1 % q + a1 * b0 % q) % q])
        c = _intt64(a1 * b1 % q, qs)
        acc = 0
        for j, (lo, hi) in enumerate(digit_ranges(L, case["alpha"])):
            rest = [k for k in range(len(qp)) if not lo <= k < hi]
            U = torch.empty((len(qp), c.shape[-1]), dtype=torch.int64, device="cuda")
            U[lo:hi] = c[lo:hi]
            U[rest] = _bconv64(c[lo:hi], qs[lo:hi], [qp[k] for k in rest])
            acc = (acc + _ntt64(U, qp) * evk[j]) % _q64(qp)
        acc = _intt64(acc, qp)
        P = 1
        for p in ps:
            P *= p
        ks = (acc[:, :L] - _bconv64(acc[:, L:], ps, qs) + q) * _q64([pow(P % v, -1, v) for v in qs]) % q
        c = _intt64((d + _ntt64(ks, qs)) % q, qs)
        ql, inv = qs[:-1], [pow(qs[-1], -1, v) for v in qs[:-1]]
        return _ntt64((c[:, :-1] - c[:, -1:] % _q64(ql) + _q64(ql)) * _q64(inv) % _q64(ql), ql)
    cts, key_q, key_p, qall, ps = _in_serve(case, seed)
    out = []
    for a0, a1, b0, b1 in [[t.long() for t in c] for c in cts]:
        qs = qall[:a0.shape[0]]
        q, p = _q64(qs), _q64(ps)
        d2 = a1 * b1 % q
        up = _ntt64(_bconv64(_intt64(d2, qs), qs, ps), ps)
        out.append(torch.cat([a0 * b0 % q, (a0 * b1 % q + a1 * b0 % q) % q] +
                             [d2 * k[:len(qs)].long() % q for k in key_q] + [up * k.long() % p for k in key_p]))
    return out
