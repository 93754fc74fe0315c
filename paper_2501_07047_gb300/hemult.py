"""HE-Mult with hybrid key switching and rescale, composed from hefx C-ABI calls.

The paper measures HE-Mult, Relin. and Rescale (Sec. V-A; dnum-digit hybrid key switching,
Sec. V-C "Effects of Security Parameters") and builds them from NTT, INTT, BConv, VecModMul
and VecModAdd (App. A); it does not print their formulas, which here are textbook RNS-CKKS:

  d0 = a0 b0, d1 = a0 b1 + a1 b0, d2 = a1 b1            tensor product (evaluation form, Q)
  c = INTT(d2) (= INTT(a1 o b1), taken from a1, b1 directly)
  per digit j (limbs D_j, alpha per digit):              ModUp
      U_j = c on D_j, BConv_{D_j -> rest of Q u P}(c) elsewhere, NTT over Q u P
  acc_k = sum_j U_j o evk_{j,k}                           key inner product
  ks_k = ModDown(INTT(acc_k)), c_k = d_k + NTT(ks_k)
  c'_k = NTT(Rescale(INTT(c_k)))                          over q_0 .. q_{L-2}

With the Rescale, INTT(c_k) = INTT(d_k) + ks_k is all that is needed of c_k, and by linearity it is
t_k - P^-1 BConv_{P->Q}(INTT(acc_k)_P) with t_k = INTT(P^-1 acc_k + d_k) over Q: the key inner product
scales and adds as it writes, and two transforms of c (NTT(ks), INTT(c), 96 limbs each at L = 48)
and the addition drop out.

Every step runs in libhefx's kernels; this module only allocates workspaces and issues the
calls on one stream.  Inputs and outputs are one ciphertext pair in evaluation form.
"""
from __future__ import annotations

from . import hefx


def digit_ranges(L: int, alpha: int):
    """Limb ranges [lo, hi) of the dnum = ceil(L / alpha) key-switching digits."""
    return [(lo, min(L, lo + alpha)) for lo in range(0, L, alpha)]


class HeMult:
    """Parameter sets, basis-conversion plans and workspaces of one shape (N, Q, P, alpha)."""

    def __init__(self, ctx: int, logn: int, qs, ps, alpha: int, ntt_path: str = "cudacore",
                 bconv_path: str = "auto"):
        import torch
        self.torch = torch
        self.ctx, self.logn = ctx, logn
        self.qs, self.ps = [int(q) for q in qs], [int(p) for p in ps]
        self.L, self.K, self.alpha = len(self.qs), len(self.ps), alpha
        if self.L < 2:
            raise ValueError("HE-Mult with rescale needs at least 2 ciphertext limbs")
        self.digits = digit_ranges(self.L, alpha)
        self.dnum = len(self.digits)
        self.ntt_path, self.bconv_path = ntt_path, bconv_path
        self.pQ = hefx.hefx_params_create(ctx, logn, self.qs)
        self.pQr = hefx.hefx_params_create(ctx, logn, self.qs[:-1])
        self.pQP = hefx.hefx_params_create(ctx, logn, self.qs + self.ps)
        qp = self.qs + self.ps
        # ModUp: one launch for every digit ("auto": on the faster path; "cudacore": on the CUDA
        # cores, and ModDown too), or two conversions per digit through hefx_basis_convert on the
        # requested path
        self.modup = hefx.hefx_modup_plan_create(ctx, logn, self.qs, self.ps, alpha) \
            if bconv_path in ("auto", "cudacore") else None
        self.plans = []
        for lo, hi in ([] if self.modup else self.digits):
            src = self.qs[lo:hi]
            lo_plan = hefx.hefx_bconv_plan_create(ctx, logn, src, self.qs[:lo]) if lo > 0 else None
            hi_plan = hefx.hefx_bconv_plan_create(ctx, logn, src, qp[hi:])
            self.plans.append((lo_plan, hi_plan))
        self.plan_pq = hefx.hefx_bconv_plan_create(ctx, logn, self.ps, self.qs)
        if bconv_path == "cudacore":
            hefx.hefx_modup_plan_set_path(ctx, self.modup, bconv_path)
            hefx.hefx_bconv_plan_set_mod_down_path(ctx, self.plan_pq, bconv_path)
        n, L, K = 1 << logn, self.L, self.K
        dev = "cuda"
        self.d = torch.empty((3, L, n), dtype=torch.int32, device=dev)
        self.c = torch.empty((L, n), dtype=torch.int32, device=dev)
        self.U = torch.empty((self.dnum, L + K, n), dtype=torch.int32, device=dev)
        self.acc = torch.empty((2, L + K, n), dtype=torch.int32, device=dev)
        self.ks = torch.empty((2, L, n), dtype=torch.int32, device=dev)
        self.cc = torch.empty((2, L, n), dtype=torch.int32, device=dev)
        self.merged = False  # the last run took the merged form (stages)

    def close(self) -> None:
        if self.modup:
            hefx.hefx_modup_plan_destroy(self.modup)
        for lo_plan, hi_plan in self.plans:
            if lo_plan:
                hefx.hefx_bconv_plan_destroy(lo_plan)
            hefx.hefx_bconv_plan_destroy(hi_plan)
        hefx.hefx_bconv_plan_destroy(self.plan_pq)
        for p in (self.pQ, self.pQr, self.pQP):
            hefx.hefx_params_destroy(p)

    def check(self, stream=None) -> None:
        """Waits for `stream` (the current one by default) and raises HefxError(ETIMEOUT) if a bounded
        device wait of an earlier run expired: of a conversion (ModUp, ModDown) or of a transform.  The
        results of those runs are invalid; the record is cleared."""
        st = self.torch.cuda.current_stream() if stream is None else stream
        checks = [(hefx.hefx_modup_check, self.modup)] if self.modup else []
        checks += [(hefx.hefx_bconv_check, p) for pair in self.plans for p in pair if p]
        checks += [(hefx.hefx_bconv_check, self.plan_pq)]
        checks += [(hefx.hefx_stream_check, p) for p in (self.pQ, self.pQr, self.pQP)]
        expired = None
        for check, handle in checks:  # all of them, so that every record is cleared
            try:
                check(self.ctx, handle, st)
            except hefx.HefxError as e:
                if e.status != hefx.HEFX_ETIMEOUT:
                    raise
                expired = expired or e
        if expired:
            raise expired

    def launches(self, rescale: bool = True, captured: bool = False) -> int:
        """Kernel launches of one run (CUDA-core NTT path), eager or captured into a graph."""
        def count(params, form, batch):
            return hefx.hefx_ntt_launches(params, form, batch, captured)

        n = 1 + count(self.pQ, "inv_hadamard", 1)  # tensor product, INTT(a1 o b1)
        n += 1 if self.modup else sum(2 if lo else 1 for lo, _ in self.digits)
        n += count(self.pQP, "fwd", self.dnum) + 1 + count(self.pQP, "inv", 2) + 1  # .., inner product, .., ModDown
        return n + (count(self.pQ, "rescale_fwd", 2) if rescale else count(self.pQ, "fwd", 2) + 1)

    def rescale_launches(self, captured: bool = False) -> int:
        """Kernel launches of rescale() (CUDA-core NTT path)."""
        return (hefx.hefx_ntt_launches(self.pQ, "inv", 2, captured) +
                hefx.hefx_ntt_launches(self.pQ, "rescale_fwd", 2, captured))

    def run(self, a0, a1, b0, b1, evk, out, stream=None, rescale: bool = True) -> None:
        """a*, b*: [L][N] evaluation form over Q; evk: [dnum][2][L+K][N] evaluation form over
        Q u P.  With rescale, out [2][L-1][N] receives (c'_0, c'_1); without, out [2][L][N]
        receives the relinearised (c_0, c_1) over Q.  Copies (c <- d2, and U_j <- c on D_j
        when ModUp runs as per-digit conversions) are device-to-device on the same stream."""
        torch = self.torch
        ctx, s = self.ctx, stream
        d0, d1, d2 = self.d[0], self.d[1], self.d[2]
        st = torch.cuda.current_stream() if s is None else s
        with torch.cuda.stream(st):
            if self.ntt_path == "cudacore":
                # d2 = a1 o b1 only feeds c = INTT(d2): the inverse transform multiplies a1 and
                # b1 as it loads them, and the tensor product writes d0 and d1 only
                hefx.hefx_tensor_product(ctx, self.pQ, a0, a1, b0, b1, d0, d1, None, 1, st)
                hefx.hefx_ntt_inv_hadamard(ctx, self.pQ, a1, b1, self.c, 1, st)
            else:
                hefx.hefx_tensor_product(ctx, self.pQ, a0, a1, b0, b1, d0, d1, d2, 1, st)
                self.c.copy_(d2)
                hefx.hefx_ntt_inv(ctx, self.pQ, self.c, 1, self.ntt_path, st)
            if self.modup:
                hefx.hefx_mod_up(ctx, self.modup, self.c, self.U, 1, st)
            for j, ((lo, hi), (lo_plan, hi_plan)) in enumerate(zip(self.digits, self.plans)):
                self.U[j, lo:hi].copy_(self.c[lo:hi])
                if lo_plan:
                    hefx.hefx_basis_convert(ctx, lo_plan, self.c[lo:hi], self.U[j, :lo], 1, self.bconv_path, st)
                hefx.hefx_basis_convert(ctx, hi_plan, self.c[lo:hi], self.U[j, hi:], 1, self.bconv_path, st)
            hefx.hefx_ntt_fwd(ctx, self.pQP, self.U, self.dnum, self.ntt_path, st)
            self.merged = rescale and self.ntt_path == "cudacore"
            if self.merged:
                hefx.hefx_key_inner_product_add(ctx, self.pQP, self.plan_pq, self.U, evk, self.d[0:2], self.acc,
                                                self.dnum, 1, st)
                hefx.hefx_ntt_inv(ctx, self.pQP, self.acc, 2, self.ntt_path, st)
                hefx.hefx_mod_down_scaled(ctx, self.plan_pq, self.acc, self.cc, 2, st)
                hefx.hefx_rescale_ntt(ctx, self.pQ, self.cc, out, 2, st)
                return
            hefx.hefx_key_inner_product(ctx, self.pQP, self.U, evk, self.acc, self.dnum, 1, st)
            hefx.hefx_ntt_inv(ctx, self.pQP, self.acc, 2, self.ntt_path, st)
            hefx.hefx_mod_down(ctx, self.plan_pq, self.acc, self.ks, 2, st)
            hefx.hefx_ntt_fwd(ctx, self.pQ, self.ks, 2, self.ntt_path, st)
            dst = self.cc if rescale else out
            # (c_0, c_1) = (d_0, d_1) + (ks_0, ks_1): both halves are contiguous, one launch
            hefx.hefx_vec_mod_add(ctx, self.pQ, self.d[0:2], self.ks, dst, 2, st)
            if rescale:
                self.rescale(self.cc, out, st)

    def rescale(self, c, out, stream=None) -> None:
        """c: [2][L][N] evaluation form over Q (overwritten) -> out [2][L-1][N] evaluation form
        over q_0 .. q_{L-2}: NTT(Rescale(INTT(c))); on the CUDA-core path the rescale runs on
        the forward transform's input load."""
        st = self.torch.cuda.current_stream() if stream is None else stream
        with self.torch.cuda.stream(st):
            hefx.hefx_ntt_inv(self.ctx, self.pQ, c, 2, self.ntt_path, st)
            if self.ntt_path == "cudacore":
                hefx.hefx_rescale_ntt(self.ctx, self.pQ, c, out, 2, st)
            else:
                hefx.hefx_rescale(self.ctx, self.pQ, c, out, 2, st)
                hefx.hefx_ntt_fwd(self.ctx, self.pQr, out, 2, self.ntt_path, st)

    def capture(self, a0, a1, b0, b1, evk, out, rescale: bool = True):
        """Records one run on fixed buffers as a CUDA graph (one graph launch replays all the
        kernel launches and copies, removing the host's per-call submission time).  A first
        eager run sets every kernel's attributes and occupancy before the capture.  Returns
        the torch.cuda.CUDAGraph; call .replay() to rerun on the same buffers."""
        torch = self.torch
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            self.run(a0, a1, b0, b1, evk, out, side, rescale)
        torch.cuda.current_stream().wait_stream(side)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            self.run(a0, a1, b0, b1, evk, out, torch.cuda.current_stream(), rescale)
        return g

    def stages(self, rescale: bool | None = None) -> dict:
        """The workspaces after a run (for stage-by-stage parity tests).  The merged form keeps
        t (P^-1 acc + d over Q, acc over P) and c in coefficient form; the stages that it does not
        compute are worked out from those here.  rescale: whether what ran last was with the Rescale
        (after a graph's replay: as it was captured); by default as the last call of run()."""
        torch = self.torch
        merged = self.merged if rescale is None else rescale and self.ntt_path == "cudacore"
        st = {"d0": self.d[0], "d1": self.d[1], "d2_coeff": self.c, "modup_eval": self.U, "c_coeff": self.cc}
        if not merged:
            return {**st, "acc_coeff": self.acc, "ks_eval": self.ks}
        s = torch.cuda.current_stream()
        q = torch.tensor(self.qs, dtype=torch.int64, device="cuda")[None, :, None]
        P = 1
        for p in self.ps:
            P *= p
        pmod = torch.tensor([P % v for v in self.qs], dtype=torch.int64, device="cuda")[None, :, None]
        d = self.d[0:2].clone()
        hefx.hefx_ntt_inv(self.ctx, self.pQ, d, 2, self.ntt_path, s)
        acc = self.acc.clone()
        acc[:, :self.L] = ((self.acc[:, :self.L].long() - d.long() + q) * pmod % q).to(torch.int32)
        ks = ((self.cc.long() - d.long() + q) % q).to(torch.int32)
        hefx.hefx_ntt_fwd(self.ctx, self.pQ, ks, 2, self.ntt_path, s)
        return {**st, "acc_coeff": acc, "ks_eval": ks}
