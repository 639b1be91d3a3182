"""The work that users of the range finder have it do, as cases that can be timed one by one.

`listed()` names twelve of them, `draw()` gives more of the same ranges.  Every case goes through the public binding
(paper_2608_28941_b200.rrf) as a program would call it.  Sizes, block sizes and tolerances are those of
paper_2608_28941_b200/workloads.py and of the tests, or generic; inputs are synthetic and made from a seed on the GPU.

A case is a dict of plain values: `op` is the call ("run", "run_colmajor", "form_q", "apply_qt", "apply_q",
"transfer"), `dtype`, `m`, `n`, `b` and, for the runs, the recipe of the singular values (`kind`, `rate`, `rank`,
`noise`), `tol`, `max_rank` and the options that change what is computed.
"""
import math

import torch

from paper_2608_28941_b200 import rrf


def listed():
    return [
        # a small dense problem in double precision, where the latency of sixteen small panels is everything
        dict(name="small_f64", op="run", dtype="f64", m=1024, n=768, b=16, kind="exp", rate=20.0, rank=512, noise=0.0,
             tol=1e-8, max_rank=256, estimator=0, fixed=False, update=True, own_buffers=True, own_omega=True),
        # an ordinary call with sizes that fit no tile and nothing allocated beforehand
        dict(name="ragged_f64", op="run", dtype="f64", m=5003, n=3001, b=64, kind="exp", rate=60.0, rank=1000, noise=0.0,
             tol=1e-4, max_rank=768, estimator=0, fixed=False, update=True, own_buffers=False, own_omega=True),
        # the fast-decaying spectrum of the stability experiment.  (Its own tolerance of 1e-13 ends in blocks sampled
        # from rounding noise, whose reflectors no two correct programs share.)
        dict(name="stress_f64", op="run", dtype="f64", m=4096, n=4096, b=32, kind="exp", rate=14.8, rank=512, noise=0.0,
             tol=1e-9, max_rank=768, estimator=0, fixed=False, update=True, own_buffers=True, own_omega=True),
        # slow algebraic decay at the size of the benchmark workload
        dict(name="large_f64", op="run", dtype="f64", m=8192, n=8192, b=64, kind="poly", rate=2.0, rank=4096, noise=0.0,
             tol=1e-4, max_rank=1024, estimator=0, fixed=False, update=True, own_buffers=True, own_omega=True),
        # the largest configuration: a tall matrix, wide blocks, rank 2048
        dict(name="largest_f64", op="run", dtype="f64", m=32768, n=16384, b=128, kind="exp", rate=150.0, rank=2560,
             noise=0.0, tol=1e-6, max_rank=2048, estimator=0, fixed=False, update=True, own_buffers=True, own_omega=True),
        # a training gradient of rank 128 plus noise in single precision, compressed up to the rank cap
        dict(name="gradient_f32", op="run", dtype="f32", m=4096, n=11008, b=64, kind="flat", rate=0.0, rank=128,
             noise=1e-3, tol=1e-2, max_rank=512, estimator=0, fixed=False, update=True, own_buffers=True, own_omega=True),
        # the same gradient with little noise: the run ends after two blocks
        dict(name="gradient_quiet_f32", op="run", dtype="f32", m=4096, n=11008, b=64, kind="flat", rate=0.0, rank=128,
             noise=1e-6, tol=1e-2, max_rank=512, estimator=0, fixed=False, update=True, own_buffers=True, own_omega=True),
        # only the basis is wanted: A stays as it is, sample vectors come from the seed, a sampled rule ends the run
        dict(name="basis_only_f64", op="run", dtype="f64", m=8192, n=8192, b=64, kind="poly", rate=2.0, rank=4096,
             noise=0.0, tol=1e-3, max_rank=512, estimator=2, fixed=False, update=False, own_buffers=True, own_omega=False),
        # column-major storage, a rank that is given beforehand
        dict(name="colmajor_f32", op="run_colmajor", dtype="f32", m=6000, n=2752, b=32, kind="exp", rate=100.0, rank=1024,
             noise=1e-4, tol=0.0, max_rank=256, estimator=0, fixed=True, update=True, own_buffers=False, own_omega=True),
        # the explicit basis after a run
        dict(name="form_q_f32", op="form_q", dtype="f32", m=4096, n=512, b=64, k=512),
        # other data projected onto the basis
        dict(name="apply_qt_f64", op="apply_qt", dtype="f64", m=8192, n=4098, b=64, k=512),
        # the state of a low-rank optimiser carried over from the last basis to the new one
        dict(name="transfer_f32", op="transfer", dtype="f32", m=4096, n=11008, b=64, k=128, k_old=256),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: any operation, sizes over the whole range (odd ones too), every block size and option."""
    f64 = rng.random() < 0.6
    op = rng.choice(["run"] * 6 + ["run_colmajor", "form_q", "apply_qt", "apply_q", "transfer"])
    b = rng.choice([16, 32, 64, 128] if f64 else [32, 64, 128])
    m, n = (max(_log(rng, 600, 14000), 6 * b) for _ in range(2))
    c = dict(op=op, dtype="f64" if f64 else "f32", m=m, n=n, b=b)
    most = min(16, min(m, n) // (2 * b))                     # blocks
    if op in ("form_q", "apply_qt", "apply_q", "transfer"):
        c["k"] = b * rng.randint(1, most)
        if op == "form_q":
            c["n"] = c["k"]
        if op == "transfer":
            c["k_old"] = b * rng.randint(1, most)
        return c
    cap = b * rng.randint(2, max(2, most))
    sampled = op == "run" and rng.random() < 0.2
    kind = rng.choice(["exp", "poly"] if f64 else ["exp", "flat"])
    rank = min(m, n, 2 * cap + b) if kind != "flat" else max(1, int(cap * rng.uniform(0.2, 0.6)))
    c.update(kind=kind, rate=round(cap * rng.uniform(0.05, 0.3), 2) if kind == "exp" else rng.choice([1.5, 2.0, 3.0]) if kind == "poly" else 0.0,
             rank=rank, noise=0.0 if f64 else rng.choice([1e-3, 1e-4, 1e-6]),
             tol=10.0 ** (rng.uniform(-7, -2) if f64 else rng.uniform(-2.5, -1)), max_rank=cap, estimator=2 if sampled else 0,
             fixed=rng.random() < 0.2, update=not (sampled and rng.random() < 0.5), own_buffers=rng.random() < 0.5,
             own_omega=rng.random() < 0.7)
    if not c["own_omega"]:
        c["n"] = n // 4 * 4                                  # the library's own sample vectors have rows of n elements
    return c


def _sigma(case, device="cpu"):
    j = torch.arange(case["rank"], dtype=torch.float64, device=device)
    if case["kind"] == "exp":
        return torch.exp(-j / case["rate"])
    if case["kind"] == "poly":
        return (j + 1.0) ** -case["rate"]
    return torch.ones_like(j)


class _Handle:
    """A library handle that is given back with the state that holds it."""

    def __init__(self):
        self.h = rrf.rrf_create(torch.cuda.current_device())

    def __del__(self):
        try:
            rrf.rrf_destroy(self.h)
        except Exception:
            pass


def _rows(rows, cols, dtype):
    """A rows x cols matrix whose rows start on 16-byte boundaries."""
    ld = -(-cols // 4) * 4
    return torch.zeros((rows, ld), dtype=dtype, device="cuda")[:, :cols]


def _matrix(case, dtype, gen):
    """Gaussian factors around the prescribed singular values, plus noise: entries of size ||sigma|| / sqrt(m n)."""
    m, n, r = case["m"], case["n"], case["rank"]
    s = _sigma(case, "cuda").to(dtype)
    u = torch.randn((m, r), generator=gen, dtype=dtype, device="cuda")
    v = torch.randn((r, n), generator=gen, dtype=dtype, device="cuda")
    full = torch.backends.cuda.matmul.allow_tf32
    torch.backends.cuda.matmul.allow_tf32 = False
    a = (u * (s / s.norm())) @ v
    torch.backends.cuda.matmul.allow_tf32 = full
    if case["noise"]:
        a += case["noise"] * math.sqrt(128.0) * torch.randn((m, n), generator=gen, dtype=dtype, device="cuda")
    return a


def _reflectors(m, k, b, dtype, gen):
    """V (m x k) and T (b x k) of the blocks of a Householder QR of a Gaussian matrix."""
    g = torch.randn((m, k), generator=gen, dtype=torch.float64, device="cuda")
    a, tau = torch.geqrf(g)
    v = torch.tril(a, -1)
    v.diagonal().fill_(1.0)
    t = torch.empty((b, k), dtype=torch.float64, device="cuda")
    for i in range(0, k, b):
        vi = v[:, i:i + b]
        t[:, i:i + b] = torch.linalg.inv(torch.triu(vi.T @ vi, 1) + torch.diag(1.0 / tau[i:i + b]))
    return v.to(dtype).contiguous(), torch.triu(t.view(b, k // b, b).transpose(0, 1)).transpose(0, 1).reshape(b, k).to(dtype).contiguous()


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    dtype = torch.float64 if case["dtype"] == "f64" else torch.float32
    st = {"case": case, "handle": _Handle(), "seed": int(seed) & 0x7FFFFFFF}
    m, n, b = case["m"], case["n"], case["b"]
    if case["op"] == "run":
        st["A"] = _rows(m, n, dtype)
        st["A"].copy_(_matrix(case, dtype, gen))
        if case["own_omega"]:
            st["omegaT"] = _rows(case["max_rank"], n, dtype)
            st["omegaT"].copy_(torch.randn((case["max_rank"], n), generator=gen, dtype=dtype, device="cuda"))
        if case["own_buffers"]:
            st["V"] = _rows(m, case["max_rank"], dtype)
            st["T"] = torch.zeros((b, case["max_rank"]), dtype=dtype, device="cuda")
            if case["update"]:
                st["B"] = _rows(case["max_rank"], n, dtype)
            p = rrf.make_params(rrf.RRF_F64 if case["dtype"] == "f64" else rrf.RRF_F32, m, n, b, case["tol"],
                                case["max_rank"], True, case["estimator"], _flags(case))
            st["workspace"] = torch.empty(rrf.rrf_workspace_bytes(p), dtype=torch.uint8, device="cuda")
    elif case["op"] == "run_colmajor":
        st["A"] = _matrix(case, dtype, gen).t().contiguous().t()
        if case["own_omega"]:
            st["omega"] = _rows(case["max_rank"], n, dtype)
            st["omega"].copy_(torch.randn((case["max_rank"], n), generator=gen, dtype=dtype, device="cuda"))
            st["omega"] = st["omega"].t()
    else:
        st["V"], st["T"] = _reflectors(m, case["k"], b, dtype, gen)
        if case["op"] == "transfer":
            st["V_old"], st["T_old"] = _reflectors(m, case["k_old"], b, dtype, gen)
            st["M"] = _rows(case["k_old"], n, dtype)
            st["M"].copy_(torch.randn((case["k_old"], n), generator=gen, dtype=dtype, device="cuda"))
        elif case["op"] != "form_q":
            st["C"] = _rows(m, n, dtype)
            st["C"].copy_(torch.randn((m, n), generator=gen, dtype=dtype, device="cuda"))
    return st


def _flags(case):
    return (rrf.RRF_FLAG_FIXED_RANK if case["fixed"] else 0) | (0 if case["update"] else rrf.RRF_FLAG_NO_UPDATE)


def run(st):
    c, h, b = st["case"], st["handle"].h, st["case"]["b"]
    if c["op"] == "run":
        r = rrf.rrf_run(h, st["A"], b, c["tol"], c["max_rank"], omegaT=st.get("omegaT"), estimator=c["estimator"],
                        flags=_flags(c), seed=st["seed"], V=st.get("V"), T=st.get("T"), B=st.get("B"),
                        workspace=st.get("workspace"))
        return _result(r)
    if c["op"] == "run_colmajor":
        return _result(rrf.rrf_run_colmajor(h, st["A"], b, c["tol"], c["max_rank"], omega=st.get("omega"),
                                            flags=_flags(c), seed=st["seed"]))
    if c["op"] == "form_q":
        return rrf.rrf_form_q(h, st["V"], st["T"], b, c["k"])
    if c["op"] == "apply_qt":
        return rrf.rrf_apply_qt(h, st["V"], st["T"], b, c["k"], st["C"])
    if c["op"] == "apply_q":
        return rrf.rrf_apply_q(h, st["V"], st["T"], b, c["k"], st["C"])
    return rrf.rrf_subspace_transfer(h, st["V_old"], st["T_old"], c["k_old"], st["V"], st["T"], c["k"], b, st["M"])


def _result(r):
    """What a run determines: columns and rows at or beyond k are left as they were."""
    out = {"k": r.k, "status": r.status, "normA2": r.normA2, "V": r.V[:, :r.k], "T": r.T[:, :r.k]}
    if r.B is not None:
        out["B"] = r.B[:r.k]
    return out


def _rank(case):
    """The least rank, in whole blocks, that can meet the tolerance (Eckart and Young), at most the cap."""
    if case["fixed"] or case["tol"] <= 0:
        return case["max_rank"]
    s2 = _sigma(case) ** 2
    total = float(s2.sum())
    floor = case["noise"] ** 2 * 128.0
    for k in range(case["b"], case["max_rank"], case["b"]):
        left = float(s2[k:].sum()) / total + floor * (1 - k / case["m"]) * (1 - k / case["n"])
        if left <= case["tol"] ** 2 * (1 + floor):
            return k
    return case["max_rank"]


def _block(y):
    """V and T of a Householder QR of y: Q = I - V T V^T."""
    a, tau = torch.geqrf(y)
    v = torch.tril(a, -1)
    v.diagonal().fill_(1.0)
    return v, torch.triu(torch.linalg.inv(torch.triu(v.T @ v, 1) + torch.diag(1.0 / tau)))


def _through(v, t, b, c, forward):
    """Q^T c (forward) or Q c, block by block, in place."""
    starts = range(0, v.shape[1], b)
    for r in starts if forward else reversed(starts):
        vi, ti = v[r:, r:r + b], t[:, r:r + b]
        c[r:] -= vi @ ((ti.T if forward else ti) @ (vi.T @ c[r:]))
    return c


def exact(case, seed):
    """What `run` returns, in 64 bits and plain torch.  A run that draws its sample vectors from the library's own
    generator has no such value here."""
    if case["op"] in ("run", "run_colmajor") and not case["own_omega"]:
        return None
    st, b = prepare(case, seed), case["b"]
    if case["op"] == "form_q":
        q = torch.eye(case["m"], case["k"], dtype=torch.float64, device="cuda")
        return _through(st["V"].double(), st["T"].double(), b, q, False)
    if case["op"] in ("apply_qt", "apply_q"):
        return _through(st["V"].double(), st["T"].double(), b, st["C"].double().clone(), case["op"] == "apply_qt")
    if case["op"] == "transfer":
        c = torch.zeros((case["m"], case["n"]), dtype=torch.float64, device="cuda")
        c[:case["k_old"]] = st["M"].double()
        c = _through(st["V_old"].double(), st["T_old"].double(), b, c, False)
        return _through(st["V"].double(), st["T"].double(), b, c, True)[:case["k"]]
    w = st["A"].double().clone()
    omega = st["omegaT"].double().t() if case["op"] == "run" else st["omega"].double()
    norm = float((w * w).sum())
    out = {"k": 0, "status": 1, "normA2": norm}
    left, vs, ts = norm, [], []
    for r in range(0, case["max_rank"], b):
        if case["estimator"] == 0 and not case["fixed"] and left <= case["tol"] ** 2 * norm:
            break
        if case["update"]:
            y = w[r:] @ omega[:, r:r + b]
        else:
            y = w @ omega[:, r:r + b]
            for i, (vi, ti) in enumerate(zip(vs, ts)):
                y[i * b:] -= vi @ (ti.T @ (vi.T @ y[i * b:]))
            y = y[r:]
        if case["estimator"] == 2:
            left = float((y * y).sum()) / b
            if not case["fixed"] and left <= case["tol"] ** 2 * norm:
                break
        v, t = _block(y)
        vs.append(v)
        ts.append(t)
        if case["update"]:
            w[r:] -= v @ (t.T @ (v.T @ w[r:]))
            if case["estimator"] == 0:
                left = float((w[r + b:] ** 2).sum())
    k = out["k"] = b * len(vs)
    out["status"] = 0 if left <= case["tol"] ** 2 * norm else 1
    out["V"] = torch.zeros((case["m"], k), dtype=torch.float64, device="cuda")
    for i, v in enumerate(vs):
        out["V"][i * b:, i * b:(i + 1) * b] = v
    out["T"] = torch.cat(ts, 1) if ts else torch.zeros((b, 0), dtype=torch.float64, device="cuda")
    if case["update"]:
        out["B"] = w[:k]
    if tolerance(case)["rel"] >= 0.03:      # the last blocks are sampled from rounding noise: any reflectors will do
        out["V"] = out["T"] = None
    return out


def work(case):
    w = 8 if case["dtype"] == "f64" else 4
    m, n, b = case["m"], case["n"], case["b"]
    if case["op"] in ("run", "run_colmajor"):
        k = _rank(case)
        size = m * n + m * k + b * k + (n * k if case["own_omega"] else 0) + (n * k if case["update"] else 0)
        if case["update"]:      # sample, V^T W and update of every block, and its panel
            flops = sum(6 * (m - r) * n * b + 3 * (m - r) * b * b for r in range(0, k, b))
        else:                   # a sample of A, all earlier reflectors on the panel, the panel
            flops = sum(2 * m * n * b + 4 * (m - r // 2) * b * r + 3 * (m - r) * b * b for r in range(0, k, b))
        return {"bytes": w * size, "flops": flops}
    k = case["k"]
    flops = sum(4 * (m - r) * n * b + 2 * n * b * b for r in range(0, k, b))
    size = m * k + b * k
    if case["op"] == "form_q":  # I[:, :k]: block column r is zero above row r, so only columns r.. are touched
        return {"bytes": w * (size + m * k), "flops": sum(4 * (m - r) * (k - r) * b for r in range(0, k, b))}
    if case["op"] == "transfer":
        ko = case["k_old"]
        flops += sum(4 * (m - r) * n * b + 2 * n * b * b for r in range(0, ko, b))
        return {"bytes": w * (size + m * ko + b * ko + ko * n + k * n), "flops": flops}
    return {"bytes": w * (size + 2 * m * n), "flops": flops}


def tolerance(case):
    """Reflectors of a late block are sampled from a residual that carries rounding noise of the size of u ||A||; two
    correct programs differ by the share this has in the residual that the last block saw, times a few (measured, one
    queue against two and the two single-precision engines against each other: 0.3 to 7), and more where the matrix's
    rank runs out inside a run, since the last panel of that rank is a square Gaussian matrix (up to 30)."""
    u = 2.2e-16 if case["dtype"] == "f64" else 6e-7
    if case["op"] in ("run", "run_colmajor"):
        s2 = _sigma(case) ** 2
        k = _rank(case)
        rest = math.sqrt(float(s2[max(0, k - case["b"]):].sum()) / float(s2.sum()) + 128.0 * case["noise"] ** 2)
        rel = 30.0 * u / min(1.0, max(rest if case["fixed"] or k == case["max_rank"] else 0.0, case["tol"], 1e-14))
        return {"rel": min(0.03, rel + (180.0 * u if case["rank"] <= k else 0.0))}
    return {"rel": (30.0 if case["dtype"] == "f64" else 15.0) * u}   # measured: 1.6e-15 and 2.1e-6
