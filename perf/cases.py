"""What the library is timed on: the calls its users make, over the sizes they make them at.

A case is one pass through a public entry point on one set of inputs:

  forward   plan.correlator(S): C of one gauge configuration (the call made most often)
  complex   mhc_correlator_cw: the same with complex wavefunction weights
  gradient  mhc.correlator under autograd, then the gradient of Re C with respect to every
            propagator and both weight vectors (the training step of a wavefunction fit)
  batch     mhc_batch_correlator: many correlators of uneven shapes in one launch
  pairs     plan.pair_dets: the per-pair determinants of a list of (source, sink) terms

Terms come in families that share all but one label per flavour (or all but two), as the
wavefunctions of the paper do; the generators are the repository's own workloads.  A term's
labels, the propagators and the weights are drawn from the seed; the family sizes are part
of the case.
"""
import math

import numpy as np
import torch

from paper_1411_3691_gb300 import mhc
from paper_1411_3691_gb300 import workloads as wl


def _L(n):
    """Label alphabet of a flavour: 12 spin-colour labels per site, one spare site."""
    return 12 * math.ceil(n / 3) + 12


def _case(kind, n, src, snk, **more):
    """n: labels per flavour, as text ("6,6").  src, snk: "FxK" (F families of K terms) or
    "ragged:N:K" (families of 1 to K terms, N terms in all)."""
    c = {"kind": kind, "n": n, "src": src, "snk": snk, "diag": 2.0, "two_row": 0.0, "forced": 0.0, "mixed": False}
    c["L"] = more.pop("L", None) or ",".join(str(_L(int(x))) for x in n.split(","))
    c.update(more)
    return c


def listed():
    return [
        # two nucleons: the smallest production call, dominated by latency and launches
        dict(_case("forward", "3,3", "64x8", "64x8", L="24,24"), name="deuteron_512"),
        # three nucleons with unequal flavours, ragged families, odd term counts
        dict(_case("forward", "5,4", "ragged:1291:16", "ragged:977:12"), name="triton_ragged"),
        # the alpha particle at the paper's 1944 terms, families of about ten
        dict(_case("forward", "6,6", "ragged:1944:20", "ragged:1944:20", L="48,48"), name="alpha_1944"),
        # He-4 at scale: the ordinary size of a measurement
        dict(_case("forward", "6,6", "256x16", "256x16", L="48,48"), name="he4_4096"),
        # the same wavefunctions with complex coefficients
        dict(_case("complex", "6,6", "128x16", "128x16", L="48,48"), name="he4_complex_2048"),
        # members of a family change rows of their own, n = 12 (Be-8-like)
        dict(_case("forward", "12,12", "128x32", "256x16", L="60,60", mixed=True), name="mixed_rows_n12"),
        # the largest single call: n = 18, two-row families, near-singular members
        dict(_case("forward", "18,18", "1024x32", "1024x32", L="96,96", diag=3.0, two_row=0.1, forced=0.01),
             name="large_nucleus"),
        # gradients: small and ragged, ordinary, and beyond the n <= 8 kernels
        dict(_case("gradient", "4,5", "ragged:515:12", "ragged:601:16"), name="triton_gradient"),
        dict(_case("gradient", "6,6", "256x16", "256x16", L="48,48"), name="he4_gradient"),
        dict(_case("gradient", "9,12", "ragged:640:24", "ragged:768:24", two_row=0.1), name="n9_n12_gradient"),
        # sixteen correlators of uneven flavours and term counts in one launch
        dict(_case("batch", "mixed", "log:256:4096:32", "log:256:4096:32", L="mixed", count=16), name="batch_16"),
        # individual determinants for a table of term pairs
        dict(_case("pairs", "18,18", "64x32", "64x32", L="96,96", diag=3.0, two_row=0.1, forced=0.01,
                   pairs=100000), name="pairs_n18"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["forward"] * 5 + ["gradient"] * 3 + ["complex", "batch", "pairs"])
    if kind == "batch":
        top = _log_int(rng, 512, 4096)
        side = "log:%d:%d:%d" % (rng.randint(64, 300), top, rng.randint(8, 32))
        return _case("batch", "mixed", side, side, L="mixed", count=rng.randint(3, 16))
    flavours = rng.choice([1] + [2] * 8 + [3])
    n = [rng.randint(3, 18 if kind != "gradient" else 14) for _ in range(flavours)]
    big = max(n)
    # term counts over the whole range, smaller for the costlier determinants
    most = (8192 if big <= 6 else 4096 if big <= 12 else 2048) // {"forward": 1, "pairs": 1}.get(kind, 2)
    sides = []
    for _ in range(2):
        k = rng.choice([1, 4, 8, 12, 16, 24, 32])
        terms = _log_int(rng, 96, most)
        sides.append("ragged:%d:%d" % (terms, k) if rng.random() < 0.7 else "%dx%d" % (max(1, terms // k), k))
    c = _case(kind, ",".join(map(str, n)), sides[0], sides[1], diag=rng.choice([2.0, 3.0]),
              two_row=rng.choice([0.0, 0.0, 0.1, 0.2]), forced=rng.choice([0.0, 0.0, 0.01]),
              mixed=rng.random() < 0.15)
    if c["mixed"]:
        c["forced"] = c["two_row"] = 0.0
    if kind == "pairs":
        c["pairs"] = _log_int(rng, 1000, 200000)
    return c


def _fams(text, rng):
    """Family sizes of a side; rng fixes the ragged ones from the case, not from the seed."""
    if text.startswith("ragged:") or text.startswith("log:"):
        p = [int(x) for x in text.split(":")[1:]]
        N = p[0] if len(p) == 2 else int(round(math.exp(rng.uniform(math.log(p[0]), math.log(p[1])))))
        sizes = []
        while sum(sizes) < N:
            sizes.append(int(rng.integers(1, p[-1] + 1)))
        sizes[-1] -= sum(sizes) - N
        return [s for s in sizes if s > 0]
    f, k = text.split("x")
    return [int(k)] * int(f)


def _shapes(case):
    """(n_f, L_f, family sizes of the source, of the sink) of each correlator of the case."""
    rng = np.random.default_rng(11)
    if case["kind"] == "batch":
        out = []
        for _ in range(case["count"]):
            n = [int(rng.choice([3, 6, 9, 12, 18])) for _ in range(2)]
            out.append((n, [_L(x) for x in n], _fams(case["src"], rng), _fams(case["snk"], rng)))
        return out
    n = [int(x) for x in case["n"].split(",")]
    return [(n, [int(x) for x in case["L"].split(",")], _fams(case["src"], rng), _fams(case["snk"], rng))]


def _workloads(case, seed):
    return [wl.make_workload("w", n, L, src, snk, diag=case["diag"], seed=[int(seed), k], two_row_frac=case["two_row"],
                             forced_frac=case["forced"], twins=8 if case["forced"] else 0, mixed_rows=case["mixed"])
            for k, (n, L, src, snk) in enumerate(_shapes(case))]


def _complex_weights(w, seed):
    rng = np.random.default_rng([int(seed), 77])
    return (w.w_src + 1j * rng.normal(size=w.w_src.shape), w.w_snk + 1j * rng.normal(size=w.w_snk.shape))


def _pair_list(case, w, seed):
    rng = np.random.default_rng([int(seed), 78])
    return (rng.integers(0, len(w.w_src), case["pairs"]), rng.integers(0, len(w.w_snk), case["pairs"]))


def prepare(case, seed):
    ws = _workloads(case, seed)
    st = {"kind": case["kind"], "plans": [mhc.Plan.from_workload(w) for w in ws],
          "S": [[torch.from_numpy(s).cuda() for s in w.S] for w in ws]}
    if case["kind"] == "complex":
        st["w"] = [torch.from_numpy(x).cuda() for x in _complex_weights(ws[0], seed)]
    elif case["kind"] == "gradient":
        st["S"] = [[s.requires_grad_(True) for s in st["S"][0]]]
        st["w"] = [torch.from_numpy(x).cuda().requires_grad_(True) for x in (ws[0].w_src, ws[0].w_snk)]
    elif case["kind"] == "batch":
        st["batch"] = _Batch(st["plans"])
        st["out"] = [torch.empty(2, dtype=torch.float64, device="cuda") for _ in ws]
    elif case["kind"] == "pairs":
        st["ij"] = [torch.from_numpy(x).cuda() for x in _pair_list(case, ws[0], seed)]
    return st


class _Batch:
    """A batch handle that is released with the state that holds it."""

    def __init__(self, plans):
        self.plans = plans  # they outlive the batch
        self.handle = mhc.mhc_batch_create([p.handle for p in plans])

    def __del__(self):
        mhc.mhc_batch_destroy(self.handle)


def run(st):
    plan, S = st["plans"][0], st["S"][0]
    if st["kind"] == "forward":
        return plan.correlator(S)
    if st["kind"] == "complex":
        return mhc.mhc_correlator_cw(plan.handle, S, *st["w"])
    if st["kind"] == "gradient":
        C = mhc.correlator(plan, S, *st["w"])
        return [C.detach(), *torch.autograd.grad(C.real, [*S, *st["w"]])]
    if st["kind"] == "pairs":
        return plan.pair_dets(S, *st["ij"])
    return mhc.mhc_batch_correlator(st["batch"].handle, st["S"], st["out"])


def work(case):
    """Bytes: propagators, labels and weights read once, results written once.  Flops: per
    (source family, sink) and flavour two triangular solves, n^2 complex multiply-adds, and the
    family's members summed against the solves, at least n_1 n_2 multiply-adds however they are
    grouped; per (source family, sink family) and flavour the LU factors of the shared block.
    A gradient takes the cofactors of the shared rows, the members' sums for both flavours and
    their scatter besides; a separate determinant takes an LU of its own."""
    total = {"bytes": 0.0, "flops": 0.0}
    for n, L, src, snk in _shapes(case):
        Ns, Nk, Fs, Fk = sum(src), sum(snk), len(src), len(snk)
        total["bytes"] += 16.0 * sum(x * x for x in L) + (Ns + Nk) * (8.0 + 4.0 * sum(n)) + 16.0
        if case["kind"] == "pairs":
            total["bytes"] += case["pairs"] * (16.0 + 16.0 * len(n))
            total["flops"] += case["pairs"] * 8.0 / 3.0 * sum(x ** 3 for x in n)
            continue
        solve = 8.0 * sum(x * x for x in n)
        sums = 8.0 * (n[0] * n[1] if len(n) > 1 else n[0])
        block = 8.0 / 3.0 * sum(x ** 3 for x in n)
        if case["kind"] == "gradient":
            total["bytes"] += 16.0 * sum(x * x for x in L) + 8.0 * (Ns + Nk)
            total["flops"] += Fs * Nk * (4.0 * solve + 2.0 * sums) + 3.0 * Fs * Fk * block
        else:
            total["flops"] += Fs * Nk * (solve + sums) + Fs * Fk * block
    return total


# ---- the same numbers from plain torch in 64 bits ---------------------------------------
def _dev():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _blocks(w, f, rows, cols):
    """The n x n matrices of flavour f for source terms `rows` x sink terms `cols`."""
    o = sum(w.n_f[:f])
    S = torch.from_numpy(w.S[f]).to(_dev())
    a = torch.from_numpy(w.labels_src[:, o:o + w.n_f[f]].astype(np.int64)).to(_dev())[rows]
    b = torch.from_numpy(w.labels_snk[:, o:o + w.n_f[f]].astype(np.int64)).to(_dev())[cols]
    return S, a, b, S[a[:, None, :, None], b[None, :, None, :]]


def _chunks(w):
    """Source terms in slices of at most about 2 GB of matrices."""
    step = max(1, int(2e9 / (16.0 * max(w.n_f) ** 2 * len(w.w_snk))))
    for i in range(0, len(w.w_src), step):
        yield torch.arange(i, min(i + step, len(w.w_src)), device=_dev())


def _matrices(w):
    return float(len(w.w_src)) * len(w.w_snk)


def _exact_C(w, ws, wk):
    cols = torch.arange(len(wk), device=_dev())
    total = torch.zeros((), dtype=torch.complex128, device=_dev())
    for rows in _chunks(w):
        p = None
        for f in range(len(w.n_f)):
            d = torch.linalg.det(_blocks(w, f, rows, cols)[3])
            p = d if p is None else p * d
        total = total + ws[rows] @ (p @ wk)
    return total


def _exact_gradient(w):
    ws, wk = (torch.from_numpy(x).to(_dev()).to(torch.complex128) for x in (w.w_src, w.w_snk))
    cols = torch.arange(len(w.w_snk), device=_dev())
    dS = [torch.zeros(s.size, dtype=torch.complex128, device=_dev()) for s in w.S]
    C = torch.zeros((), dtype=torch.complex128, device=_dev())
    dws, dwk = torch.zeros_like(ws), torch.zeros_like(wk)
    for rows in _chunks(w):
        dets, labels, cof = [], [], []
        for f in range(len(w.n_f)):
            S, a, b, G = _blocks(w, f, rows, cols)
            d = torch.linalg.det(G)
            dets.append(d)
            cof.append(d[..., None, None] * torch.linalg.inv(G).transpose(-1, -2))
            labels.append((a[:, None, :, None] * S.shape[0] + b[None, :, None, :]).expand(G.shape))
            del G
        p = math.prod(dets[1:], start=dets[0])
        C += ws[rows] @ (p @ wk)
        dws[rows] = p @ wk
        dwk += ws[rows] @ p
        for f in range(len(w.n_f)):
            g = ws[rows][:, None] * wk[None, :]
            for k in range(len(w.n_f)):
                if k != f:
                    g = g * dets[k]
            dS[f].index_add_(0, labels[f].reshape(-1), (g[..., None, None] * cof[f]).reshape(-1))
    # torch's gradient of the real loss Re C is conj(dC/dS)
    return [C, *[x.conj().reshape(s.shape).resolve_conj() for x, s in zip(dS, w.S)], dws.real.contiguous(),
            dwk.real.contiguous()]


def exact(case, seed):
    ws = _workloads(case, seed)
    size = sum(_matrices(w) * sum(x ** 3 for x in w.n_f) for w in ws)
    if case["kind"] == "pairs":
        ii, jj = (torch.from_numpy(x) for x in _pair_list(case, ws[0], seed))
        out = []
        for f, n in enumerate(ws[0].n_f):
            o = sum(ws[0].n_f[:f])
            a = torch.from_numpy(ws[0].labels_src[:, o:o + n].astype(np.int64))[ii]
            b = torch.from_numpy(ws[0].labels_snk[:, o:o + n].astype(np.int64))[jj]
            out.append(torch.linalg.det(torch.from_numpy(ws[0].S[f])[a[:, :, None], b[:, None, :]].to(_dev())))
        return torch.stack(out, dim=1)
    if case["kind"] == "gradient":
        return _exact_gradient(ws[0]) if size < 1.2e10 else None
    if size > 6e10:
        return None
    if case["kind"] == "complex":
        C = _exact_C(ws[0], *(torch.from_numpy(x).to(_dev()) for x in _complex_weights(ws[0], seed)))
        return torch.view_as_real(C)
    out = [torch.view_as_real(_exact_C(w, *(torch.from_numpy(x).to(_dev()).to(torch.complex128)
                                            for x in (w.w_src, w.w_snk)))) for w in ws]
    return out if case["kind"] == "batch" else out[0]
