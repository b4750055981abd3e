"""The work that users of this library have it do, as timed cases over its real range of sizes.

A case is one pass through the public entry points: a solve of a book of accounts (from host or
device buffers, in each precision that is used in earnest), a training step through the autograd
function, or the allocation-free polish of weights that the caller already holds. Sizes are those
of the workload generator, the tests and the benchmark; `draw` spreads over the same ranges.

`exact` solves the books without a turnover cap and tax lots again in plain torch and numpy: a
splitting iteration in FP32 finds the active set, a dense FP64 solve of the optimality conditions
on it gives the values, and every condition is checked in FP64 before they are handed out.
"""
import math

import numpy as np
import torch

from paper_2606_23367_gb300 import autograd, prism
from paper_2606_23367_gb300.workloads import Batch, loss_weights, make_workload

PRECISION = {"plain64": prism.PRISM_PLAIN_FP64, "plain32": prism.PRISM_PLAIN_FP32,
             "fp32": prism.PRISM_BATCHED_FP32, "bf16": prism.PRISM_BATCHED_BF16}
FACTOR_WIDTH = 0.03                # the constraint-burden bundles' factor-exposure bounds


def _case(kind, workload, N, K, M, precision="bf16", host=False, factor_rows=0, tilt=0.0, bench=False, **more):
    return dict(kind=kind, workload=workload, N=N, K=K, M=M, precision=precision, host=host,
                factor_rows=factor_rows, tilt=tilt, bench=bench, **more)


def listed():
    return [
        # one account rebalanced on request, all in host memory: the latency of a call, in the
        # reference precision and in the default one
        _case("solve", 0, 100, 10, 1, "plain64", host=True, name="single_100_plain64"),
        _case("solve", 0, 100, 10, 1, "bf16", host=True, name="single_100_bf16"),
        # a desk's small book, sizes that are multiples of nothing
        _case("solve", 1, 777, 17, 37, name="book_37x777"),
        # the FP32 mode on a book of ordinary size
        _case("solve", 1, 5000, 48, 128, "fp32", name="book_128x5000_fp32"),
        # one micro-batch of the production queue: host buffers in, host buffers out
        _case("solve", 1, 10000, 64, 100, host=True, name="queue_100x10000_host"),
        # the headline book, resident on the device
        _case("solve", 1, 10000, 64, 500, name="book_500x10000"),
        # accounts of 100 to 5,000 names each
        _case("solve", 2, 5000, 32, 256, name="ragged_256x5000"),
        # taxable accounts: lots, restriction caps, a turnover cap
        _case("solve", 3, 1924, 48, 200, name="tax_200x1924"),
        # a mandate with a benchmark, a view (tilt) and factor-exposure bounds
        _case("solve", 4, 2000, 32, 64, factor_rows=4, tilt=0.01, bench=True, name="mandate_64x2000"),
        # a training step: the risk model comes fresh from a network, weights forward, gradients back
        _case("train", 4, 2000, 32, 128, name="train_128x2000"),
        # yesterday's weights polished and certified without allocating
        _case("warm", 4, 2000, 32, 8, name="warm_8x2000"),
    ]


def _log(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["single", "book", "book", "queue", "ragged", "tax", "mandate", "train", "warm"])
    if kind == "single":
        return _case("solve", 0, _log(rng, 60, 400), rng.randint(4, 16), 1, rng.choice(["plain64", "plain32", "bf16"]),
                     host=True)
    if kind == "book":
        return _case("solve", 1, _log(rng, 700, 10000), rng.randint(8, 64), _log(rng, 4, 500),
                     rng.choice(["bf16", "bf16", "fp32"]))
    if kind == "queue":
        return _case("solve", 1, _log(rng, 2000, 10000), rng.randint(16, 64), _log(rng, 10, 100), host=True)
    if kind == "ragged":
        return _case("solve", 2, _log(rng, 900, 5000), rng.randint(12, 32), _log(rng, 4, 256))
    if kind == "tax":
        return _case("solve", 3, _log(rng, 400, 1924), rng.randint(12, 48), _log(rng, 4, 200))
    if kind == "mandate":
        return _case("solve", 4, _log(rng, 900, 2000), rng.randint(12, 32), _log(rng, 4, 64), factor_rows=rng.randint(0, 4),
                     tilt=rng.choice([0.0, 0.01]), bench=True)
    if kind == "train":
        return _case("train", 4, _log(rng, 500, 2000), rng.randint(8, 32), _log(rng, 2, 128))
    n = _log(rng, 500, 4000)
    return _case("warm", 4, n, rng.randint(8, 32), min(_log(rng, 1, 32), 131072 // (-(-n // 64) * 64)))


# ---------------------------------------------------------------------------
# inputs and passes
# ---------------------------------------------------------------------------
def _book(case, seed):
    over = dict(N=case["N"], K=case["K"], M=case["M"])
    if case["factor_rows"]:
        over["factor_bound"] = (case["factor_rows"], FACTOR_WIDTH)
    if case["tilt"]:
        over["tilt"] = case["tilt"]
    if case["bench"]:
        over["bench"] = True
    if case["workload"] != 2:
        return make_workload(case["workload"], seed=seed, **over)
    # accounts of 100 to N names, evenly over the logarithm and in no order; the sizes do not depend
    # on the seed, so that outputs of two seeds have one shape
    sizes = np.random.default_rng(0).permutation(np.geomspace(100, case["N"], case["M"]).round().astype(int))
    books = [make_workload(2, seed=seed, first_account=a, ragged=(int(n), int(n)), **{**over, "M": 1})
             for a, n in enumerate(sizes)]
    batches = [b for _, b in books]
    joined = {k: np.concatenate([getattr(b, k) for b in batches])
              for k in ("asset_idx", "w0", "lower", "upper", "tc", "band_lo", "band_hi", "turnover_cap")}
    return books[0][0], Batch(offsets=np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64), **joined)


def _dev(x):
    return None if x is None else torch.from_numpy(np.ascontiguousarray(x)).cuda()


BOOK_ARRAYS = ("offsets", "asset_idx", "w0", "lower", "upper", "tc", "band_lo", "band_hi", "turnover_cap",
               "lot_offsets", "lot_size", "lot_kappa", "mu_tilt", "w_bench", "factor_lo", "factor_hi")


def _outputs(M, S, K, nnz):
    z = lambda *shape: torch.zeros(*shape, dtype=torch.float64, device="cuda")  # noqa: E731
    return dict(w=z(nnz), status=torch.zeros(M, dtype=torch.int32).pin_memory(), iters=None, nu=z(M),
                lambda_band=z(M, S), theta=z(M), diag=z(M, prism.PRISM_NDIAG), kappa=z(M, K))


def prepare(case, seed):
    uni, batch = _book(case, seed)
    M, S, K, nnz = batch.n_accounts, uni.n_sectors, uni.n_factors, int(batch.offsets[-1])
    state = dict(case=case)
    if case["kind"] == "train":
        state["risk"] = [_dev(x) for x in (uni.mu, uni.B, uni.d, batch.w0)]
        state["spec"] = dict(f=_dev(uni.f), sector=_dev(uni.sector), n_sectors=S,
                             **{k: _dev(getattr(batch, k)) for k in ("offsets", "lower", "upper", "tc", "band_lo",
                                                                     "band_hi", "turnover_cap")})
        state["g"] = _dev(loss_weights(case["workload"], batch, seed))
        return state
    state["universe"] = prism.create_universe(uni)
    if case["host"]:
        state["batch"] = batch
        return state
    state["book"] = {k: _dev(getattr(batch, k)) for k in BOOK_ARRAYS}
    state["out"] = _outputs(M, S, K, nnz)
    if case["kind"] == "warm":
        # weights of an earlier solve, drifted a little since (the entry takes a start within 1e-4
        # of the band edges)
        w = prism.solve(state["universe"], batch)["w"]
        r = np.random.default_rng([seed, 1])
        inside = (w > batch.lower + 1e-12) & (w < batch.upper - 1e-12) & (np.abs(w - batch.w0) > 1e-12)
        w = np.clip(w * (1.0 + 1e-4 * r.uniform(-1.0, 1.0, size=w.shape) * inside), batch.lower, batch.upper)
        state["w_in"] = _dev(w)
        state["book"] = {k: state["book"][k] for k in BOOK_ARRAYS[:9]}
        del state["out"]["kappa"]
    return state


def _returned(r, case):
    """What a solve returns. Of the diagnostics, the last column (a bound formed from residuals at the
    level of FP64 rounding) has no value of its own to compare; the other residuals stand beside
    the objective that they certify. Iteration counts are not results."""
    out = {k: r[k] for k in ("w", "status", "nu", "lambda_band", "theta")}
    out["diag"] = r["diag"][:, :prism.PRISM_DIAG_ERR_EST]
    if case["factor_rows"]:
        out["kappa"] = r["kappa"]
    return out


def run(state):
    case = state["case"]
    if case["kind"] == "train":
        mu, B, d, w0 = (t.clone().requires_grad_() for t in state["risk"])   # a network's output tensors
        w = autograd.solve(mu, B, d, w0, **state["spec"])
        return dict(zip(("w", "dmu", "dB", "dd", "dw0"),
                        (w.detach(), *torch.autograd.grad(w, (mu, B, d, w0), state["g"]))))
    stream = torch.cuda.current_stream().cuda_stream
    if case["kind"] == "warm":
        return _returned(prism.prism_polish_noalloc(state["universe"], w_in=state["w_in"], out=state["out"],
                                                    cuda_stream=stream, **state["book"]), case)
    if case["host"]:
        return _returned(prism.solve(state["universe"], state["batch"], precision=PRECISION[case["precision"]]), case)
    return _returned(prism.prism_solve_batch(state["universe"], out=state["out"], cuda_stream=stream,
                                             precision=PRECISION[case["precision"]], **state["book"]), case)


def work(case):
    """Each input read once and each output written once, and the arithmetic of one gradient of the
    risk term per account (the product with B' and the one with B): what any method has to do."""
    N, K, M = case["N"], case["K"], case["M"]
    names = M * N
    if case["workload"] == 2:          # 100 to N names an account, evenly over their logarithm
        names = M * (N - 100) / math.log(N / 100)
    arrays = 5 + bool(case["tilt"]) + case["bench"] + 0.5 * (case["workload"] == 2) + 2.5 * (case["workload"] == 3)
    if case["kind"] == "train":
        arrays += 2                    # the gradient of the loss in, the one of the holdings out
    if case["kind"] == "warm":
        arrays += 1
    model = (2 if case["kind"] == "train" else 1) * 8.0 * N * (K + 2)
    return {"bytes": 8.0 * arrays * names + model, "flops": 4.0 * names * K * (2 if case["kind"] == "train" else 1)}


# ---------------------------------------------------------------------------
# the same values from plain torch and numpy
# ---------------------------------------------------------------------------
def _dense(x, offs, idx, M, N):
    out = np.zeros((M, N))
    for a in range(M):
        out[a, slice(None) if idx is None else idx[offs[a]:offs[a + 1]]] = x[offs[a]:offs[a + 1]]
    return out


def _iterate(B, f, d, m, sector, S, l, u, w0, c, lo, hi, flo, fhi, steps, rho=3.0):
    """A splitting iteration over all accounts (FP32): the point z and which bands and factor bounds
    hold it. The projection onto budget and bands finds its multipliers by bisection."""
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    t = lambda x: torch.as_tensor(np.ascontiguousarray(x), dtype=torch.float32, device=dev)  # noqa: E731
    Bt, m, l, u, w0, c, lo, hi = (t(x) for x in (B, m, l, u, w0, c, lo, hi))
    rows = np.flatnonzero(np.isfinite(flo).any(0) | np.isfinite(fhi).any(0))
    g = 2.0 * f
    g[rows] += rho
    D = 2.0 * d + rho
    C = np.linalg.inv(np.diag(1.0 / g) + B.T @ (B / D[:, None]))
    C, Di, Br, flo, fhi = t(C), t(1.0 / D), Bt[:, rows], t(flo[:, rows]), t(fhi[:, rows])
    hot = torch.zeros(B.shape[0], S, dtype=torch.float32, device=dev)
    sec = torch.as_tensor(sector.astype(np.int64), device=dev)
    hot[torch.arange(B.shape[0], device=dev), sec] = 1.0
    z = w0.clamp(min=l, max=u)
    y = torch.zeros_like(z)
    s = torch.zeros_like(flo)
    ys = torch.zeros_like(s)
    k = c / rho

    def prox(v, eta):
        q = v - eta / rho - w0
        return (w0 + q.sign() * (q.abs() - k).clamp(min=0)).clamp(min=l, max=u)

    for _ in range(steps):
        r = (m + rho * (z - y) + (rho * (s - ys)) @ Br.T) * Di
        x = r - (((r @ Bt) @ C) @ Bt.T) * Di
        v = x + y
        e0 = (rho * (v - u).amin(1) - c.amax(1))[:, None]
        e1 = (rho * (v - l).amax(1) + c.amax(1))[:, None]

        def root(above, shape):
            a, b = e0.expand(shape).clone(), e1.expand(shape).clone()
            for _ in range(36):
                mid = 0.5 * (a + b)
                up = above(mid)
                a, b = torch.where(up, mid, a), torch.where(up, b, mid)
            return 0.5 * (a + b)

        at = lambda eta: prox(v, eta[:, sec]) @ hot  # noqa: E731
        shape = (z.shape[0], S)
        eta_hi = torch.where(torch.isfinite(hi), root(lambda e: at(e) > hi, shape), e0 - 1.0)
        eta_lo = torch.where(lo > 0, root(lambda e: at(e) >= lo, shape), e1 + 1.0)
        clip = lambda e: torch.minimum(torch.maximum(e.expand(shape), eta_hi), eta_lo)  # noqa: E731
        nu = root(lambda e: at(clip(e)).sum(1, keepdim=True) > 1.0, (z.shape[0], 1))
        z = prox(v, clip(nu)[:, sec])
        y = v - z
        ex = x @ Br
        s = torch.minimum(torch.maximum(ex + ys, flo), fhi)
        ys = ex + ys - s
    wb = (eta_hi > nu).int() - (eta_lo < nu).int()
    wf = np.zeros((z.shape[0], B.shape[1]), np.int64)
    wf[:, rows] = ((s == fhi).int() - (s == flo).int()).cpu().numpy()
    return z.cpu().numpy(), wb.cpu().numpy(), wf


LOWER, HELD, UPPER, BELOW, ABOVE = range(5)     # on l, on w0, on u; between l and w0, between w0 and u


def _settle(B, f, d, m, sector, l, u, w0, c, lo, hi, flo, fhi, z, wb, wf):
    """One account: the optimality conditions solved in FP64 on an active set, which is corrected until
    all of them hold. None if it does not come to that."""
    inner = (w0 > l) & (w0 < u)
    side = np.where(w0 <= l, ABOVE, BELOW)      # where w0 is no inner kink, the one segment there is
    l32, u32, w32 = (x.astype(np.float32) for x in (l, u, w0))
    st = np.where(inner, np.where(z < w32, BELOW, ABOVE), side)
    st = np.where(inner & (z == w32), HELD, np.where(z == u32, UPPER, st))
    st = np.where((z == l32) | (u <= l), LOWER, st)
    wb, wf = wb.copy(), wf.copy()
    top = {BELOW: np.where(inner, w0, u), ABOVE: u}
    low = {BELOW: l, ABOVE: np.where(inner, w0, l)}
    for _ in range(100):
        F = st >= BELOW
        w = np.where(st == LOWER, l, np.where(st == HELD, w0, np.where(st == UPPER, u, 0.0)))
        bands, facs = np.flatnonzero(wb), np.flatnonzero(wf)
        E = np.concatenate([np.ones((1, w.size)), (sector[None] == bands[:, None]).astype(float), B[:, facs].T])
        e = np.concatenate([[1.0], np.where(wb > 0, hi, lo)[bands], np.where(wf > 0, fhi, flo)[facs]])
        n, r = int(F.sum()), len(e)
        KKT = np.zeros((n + r, n + r))
        KKT[:n, :n] = 2.0 * (B[F] * f) @ B[F].T + np.diag(2.0 * d[F])
        KKT[:n, n:], KKT[n:, :n] = E[:, F].T, E[:, F]
        slope = np.where(st == ABOVE, c, -c)
        rhs = np.concatenate([(m - slope - 2.0 * (B @ (f * (B.T @ w))))[F], e - E @ w])
        try:
            x = np.linalg.solve(KKT, rhs)
            x += np.linalg.solve(KKT, rhs - KKT @ x)
        except np.linalg.LinAlgError:
            return None
        w[F] = x[:n]
        nu, lam, kappa = x[n], np.zeros(len(wb)), np.zeros(len(wf))
        lam[bands], kappa[facs] = x[n + 1:n + 1 + len(bands)], x[n + 1 + len(bands):]
        h = B.T @ w
        pull = -(2.0 * (B @ (f * h) + d * w) - m + nu + lam[sector] + B @ kappa)
        new = st.copy()
        for seg in (BELOW, ABOVE):
            new[(st == seg) & (w > top[seg] + 1e-12)] = HELD if seg == BELOW else UPPER
            new[(st == seg) & (w < low[seg] - 1e-12)] = LOWER if seg == BELOW else HELD
        new[(new == HELD) & ~inner & (st == BELOW)] = UPPER
        new[(new == HELD) & ~inner & (st == ABOVE)] = LOWER
        out = np.where(side == ABOVE, c, -c)
        ends = u > l
        new[(st == LOWER) & ends & (pull > np.where(inner, -c, out) + 1e-11)] = BELOW
        new[(st == UPPER) & ends & (pull < np.where(inner, c, out) - 1e-11)] = ABOVE
        new = np.where((new >= BELOW) & (st < BELOW) & ~inner, side, new)
        new[(st == HELD) & (pull > c + 1e-11)] = ABOVE
        new[(st == HELD) & (pull < -c - 1e-11)] = BELOW
        sums = np.bincount(sector, w, len(wb))
        wb2 = np.where((wb > 0) & (lam < -1e-11) | (wb < 0) & (lam > 1e-11), 0, wb)
        wb2 = np.where(wb == 0, (sums > hi + 1e-12).astype(int) - (sums < lo - 1e-12), wb2)
        wf2 = np.where((wf > 0) & (kappa < -1e-11) | (wf < 0) & (kappa > 1e-11), 0, wf)
        wf2 = np.where(wf == 0, (h > fhi + 1e-12).astype(int) - (h < flo - 1e-12), wf2)
        if np.array_equal(new, st) and np.array_equal(wb2, wb) and np.array_equal(wf2, wf):
            obj = h @ (f * h) + w @ (d * w) - m @ w + np.abs(w - w0) @ c
            return dict(w=w, nu=nu, lam=lam, kappa=kappa, obj=obj, F=F, E=E, KKT=KKT, held=st == HELD, h=h)
        st, wb, wf = new, wb2, wf2
    return None


def exact(case, seed):
    if case["workload"] == 3:          # the cap and the lots' kinks would take a splitting of their own, many times as long
        return None
    uni, b = _book(case, seed)
    N, K, M, S = uni.n_assets, uni.n_factors, b.n_accounts, uni.n_sectors
    offs, idx = b.offsets, b.asset_idx
    l, u, w0, c, tilt = (_dense(np.zeros(int(offs[-1])) if x is None else x, offs, idx, M, N)
                         for x in (b.lower, b.upper, b.w0, b.tc, b.mu_tilt))
    m = uni.mu[None] + tilt
    if b.w_bench is not None:
        wb = _dense(b.w_bench, offs, idx, M, N)
        m = m + 2.0 * (((wb @ uni.B) * uni.f) @ uni.B.T + wb * uni.d)
    flo = np.full((M, K), -np.inf) if b.factor_lo is None else b.factor_lo
    fhi = np.full((M, K), np.inf) if b.factor_hi is None else b.factor_hi
    got, left = [None] * M, np.arange(M)
    for steps in (160, 1500):              # the few accounts whose active set the first leaves unclear once more, for longer
        z, wband, wfac = _iterate(uni.B, uni.f, uni.d, m[left], uni.sector, S, l[left], u[left], w0[left], c[left],
                                  b.band_lo[left], b.band_hi[left], flo[left], fhi[left], steps)
        for k, a in enumerate(left):
            i = np.arange(N) if idx is None else idx[offs[a]:offs[a + 1]].astype(np.int64)
            got[a] = _settle(uni.B[i], uni.f, uni.d[i], m[a, i], uni.sector[i], l[a, i], u[a, i], w0[a, i], c[a, i],
                             b.band_lo[a], b.band_hi[a], flo[a], fhi[a], z[k, i], wband[k], wfac[k])
        left = np.array([a for a in left if got[a] is None], dtype=np.int64)
        if not len(left):
            break
    else:
        return None
    w = np.concatenate([r["w"] for r in got])
    if case["kind"] == "train":
        # the optimality conditions on the active set, differentiated
        g = loss_weights(case["workload"], b, seed).reshape(M, N)
        dmu, dB, dd, dw0 = np.zeros(N), np.zeros((N, K)), np.zeros(N), np.zeros((M, N))
        for a, r in enumerate(got):
            n = int(r["F"].sum())
            x = np.linalg.solve(r["KKT"], np.concatenate([g[a, r["F"]], np.zeros(len(r["KKT"]) - n)]))
            v = np.zeros(N)
            v[r["F"]] = x[:n]
            t = uni.B.T @ v
            dmu += v
            dd -= 2.0 * r["w"] * v
            dB -= 2.0 * (np.outer(v, uni.f * r["h"]) + np.outer(r["w"], uni.f * t))
            moved = g[a] - 2.0 * (uni.B @ (uni.f * t)) - r["E"].T @ x[n:]
            dw0[a, r["held"]] = moved[r["held"]]
        return dict(w=w, dmu=dmu, dB=dB, dd=dd, dw0=dw0.reshape(-1))
    diag = np.zeros((M, prism.PRISM_DIAG_ERR_EST))
    diag[:, prism.PRISM_DIAG_OBJ] = [r["obj"] for r in got]
    out = dict(w=w, status=None, nu=np.array([r["nu"] for r in got]), lambda_band=np.stack([r["lam"] for r in got]),
               theta=np.zeros(M), diag=diag)
    if case["factor_rows"]:
        out["kappa"] = np.stack([r["kappa"] for r in got])
    return out
