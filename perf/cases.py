"""The work that a user of this library has it do, as measurable cases.

``listed()`` holds the named cases, ``draw(rng)`` one more of the same ranges;
``prepare`` makes what a program has in hand before the call, ``run`` is one
pass through the public entry points, ``work`` the bytes and operations that
the pass cannot do without, and ``exact`` the same outputs in 64 bits, by plain
torch and without this library.

Fields of a case: ``kind`` (one of KINDS), ``L`` and ``B`` (lattice and block
extents, "x.y.z.t"), ``ntv``, ``nrhs``, ``prec`` ("fp64", "fp32", "fp16": FP16
links with FP32 vectors, "bf16"), ``eps`` (spread of the links) and per kind the
solver's parameters.  A batch lists its lattices as "L/ntv/nrhs/prec/eps" joined by
spaces, all with 4^4 blocks.
"""
import math

import torch

import paper_1512_04506_gb300 as amg

M0, CSW = -0.3, 1.0
C128, C64 = torch.complex128, torch.complex64
KINDS = ("cgc", "cgc_eo", "mixed", "batch", "vcycle", "dirac", "setup")
PREC = {"fp64": amg.AMG_FP64, "fp32": amg.AMG_FP32, "fp16": amg.AMG_FP16_SCALED, "bf16": amg.AMG_BF16}


def _case(kind, L, B, ntv, nrhs, prec, eps=0.3, name=None, **more):
    c = {"kind": kind, "L": ".".join(map(str, L)), "B": ".".join(map(str, B)), "ntv": ntv, "nrhs": nrhs,
         "prec": prec, "eps": eps}
    if kind in ("cgc", "cgc_eo", "vcycle"):
        c.update(tol=0.05, restart=30, max_applies=200)  # Alg. 2's coarse solve: a residual of about 0.05
    if kind == "vcycle":
        c.update(n_smoother=4, n_mr=4)
    c.update(more)
    if name:
        c["name"] = name
    return c


def listed():
    b4 = (4, 4, 4, 4)
    return [
        # the smallest call: one correction on a 4^4 lattice in doubles, all launches and latency
        _case("cgc", (4, 4, 4, 4), (2, 2, 2, 2), 8, 1, "fp64", name="cgc_4_fp64"),
        # the coarse-grid correction of Alg. 2 as a preconditioner calls it, one right-hand side
        _case("cgc", (32, 32, 32, 32), b4, 20, 1, "fp32", name="cgc_32_fp32"),
        # the even/odd coarse solve of Alg. 2 for a block of sources (several right-hand sides)
        _case("cgc_eo", (24, 24, 24, 48), b4, 20, 8, "fp32", name="cgc_eo_24x48_fp32_8rhs"),
        # many right-hand sides on the tensor cores: BF16 storage, one propagator's worth of sources
        _case("cgc", (24, 24, 24, 48), b4, 24, 16, "bf16", name="cgc_24x48_bf16_16rhs"),
        # the batched mixed-precision coarse solve to 1e-4: FP16 links inside, FP32 refinement outside
        _case("mixed", (24, 24, 24, 48), b4, 24, 16, "fp16", name="mixed_24x48_fp16_16rhs", tol=1e-4, inner_tol=0.05,
              restart=30, max_applies=200),
        # several lattices of uneven size in one launch, as a server of small and large problems has them
        {"kind": "batch", "name": "batch_uneven", "lattices": "16.16.16.16/16/1/fp32/0.2 24.24.24.48/20/4/bf16/0.3 "
                                                              "32.32.32.64/24/12/bf16/0.4"},
        # Alg. 1, the preconditioner of the outer solve: the correction, then the smoother; one source
        _case("vcycle", (32, 32, 32, 32), b4, 20, 1, "fp32", name="vcycle_32_fp32"),
        # the same for a block of columns, as the adaptive setup sends its test vectors through it
        _case("vcycle", (16, 16, 16, 32), b4, 24, 12, "fp32", name="vcycle_16x32_fp32_12rhs"),
        # double precision, uneven extents and blocks, an odd number of test vectors and of columns
        _case("vcycle", (12, 8, 24, 16), (3, 4, 4, 2), 11, 3, "fp64", name="vcycle_ragged_fp64_3rhs"),
        # the fine operator alone: the residual and the Krylov step of the outer solver
        _case("dirac", (32, 32, 32, 64), b4, 20, 1, "fp32", name="dirac_32x64_fp32"),
        # the setup of Alg. 5, rebuilt for every gauge configuration; arithmetic in pairs of FP32 numbers
        _case("setup", (16, 16, 16, 32), b4, 24, 16, "fp32", name="setup_16x32_pair", arith="pair"),
        # the same in the default arithmetic (doubles)
        _case("setup", (16, 16, 16, 16), b4, 20, 1, "fp32", name="setup_16_fp64", arith="fp64"),
    ]


# ------------------------------------------------------------------ drawn cases
_BLOCKS = [(4, 4, 4, 4), (4, 4, 4, 4), (2, 2, 2, 2), (2, 4, 4, 4), (4, 4, 4, 2), (3, 3, 3, 3), (3, 4, 4, 2), (2, 2, 4, 4)]


def _lattice(rng, B, lo, hi, even):
    """Extents that B divides, coarse extents >= 2 (even when asked), about lo .. hi sites."""
    want = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    best = None
    for _ in range(200):
        Lc = [2 * rng.randint(1, 8) if even else rng.randint(2, 16) for _ in range(4)]
        if max(Lc) > 4 * min(Lc):
            continue
        L = [c * b for c, b in zip(Lc, B)]
        off = abs(math.log(math.prod(L) / want))
        if math.prod(L) <= hi and (best is None or off < best[0]):
            best = (off, L)
    return tuple(best[1]) if best else tuple(2 * b for b in B)


def draw(rng):
    kind = rng.choice(KINDS)
    eps = round(rng.uniform(0.2, 0.4), 3)
    if kind == "batch":
        out = []
        for _ in range(rng.randint(2, 3)):
            L = _lattice(rng, (4, 4, 4, 4), 4096, 700000, False)
            prec = rng.choice(["fp32", "bf16"])
            nrhs = rng.choice([4, 8, 12, 16]) if prec == "bf16" else rng.randint(1, 4)
            out.append("%s/%d/%d/%s/%g" % (".".join(map(str, L)), rng.choice([8, 12, 16, 20, 24]), nrhs, prec, eps))
        return {"kind": "batch", "lattices": " ".join(out)}
    B = rng.choice(_BLOCKS)
    top = 6 * math.prod(B)
    if kind in ("cgc", "cgc_eo", "vcycle"):
        prec = rng.choice(["fp64", "fp32", "fp32"] + (["bf16", "bf16"] if kind == "cgc" else []))
        if prec == "bf16":
            B, top = (4, 4, 4, 4), 1536
        nrhs = rng.choice([4, 8, 12, 16]) if prec == "bf16" else rng.choice([1, 1, 2, 3, 4, 5, 8, 11, 16])
        hi = {"fp64": 150000, "fp32": 700000, "bf16": 500000}[prec] // (1 if nrhs <= 4 else 4)
        L = _lattice(rng, B, 256 if prec == "fp64" else 4096, hi, kind != "cgc")
        ntv = rng.choice([8, 12, 16, 20, 24] if prec == "bf16" else [4, 6, 7, 8, 11, 16, 20, 24])
        return _case(kind, L, B, min(ntv, top), nrhs, prec, eps)
    if kind == "mixed":
        L = _lattice(rng, (4, 4, 4, 4), 4096, 600000, False)
        return _case(kind, L, (4, 4, 4, 4), rng.choice([8, 12, 16, 20, 24]), rng.choice([4, 8, 12, 16]), "fp16", eps,
                     tol=1e-4, inner_tol=0.05, restart=30, max_applies=200)
    if kind == "dirac":
        prec = rng.choice(["fp64", "fp32", "fp32"])
        nrhs = rng.choice([1, 1, 2, 3, 4, 7, 12])
        L = _lattice(rng, B, 4096, 2000000 // (nrhs if prec == "fp32" else 4 * nrhs), False)
        return _case(kind, L, B, 4, nrhs, prec, eps)
    arith = rng.choice(["pair", "fp64"])
    L = _lattice(rng, B, 256, 130000 if arith == "pair" else 40000, False)
    return _case("setup", L, B, min(rng.choice([6, 8, 11, 16, 20, 24]), top), rng.choice([1, 4, 16]), "fp32", eps,
                 arith=arith)


# ------------------------------------------------------------------ inputs
def _dims(text):
    return tuple(int(v) for v in text.split("."))


def _parts(case):
    """The lattices of a case as dicts (one unless it is a batch)."""
    if case["kind"] != "batch":
        return [dict(case, L=_dims(case["L"]), B=_dims(case["B"]))]
    out = []
    for item in case["lattices"].split():
        L, ntv, nrhs, prec, eps = item.split("/")
        out.append({"kind": "batch", "L": _dims(L), "B": (4, 4, 4, 4), "ntv": int(ntv), "nrhs": int(nrhs), "prec": prec,
                    "eps": float(eps)})
    return out


def _mm3(a, b):
    """Product of stacks of 3x3 matrices."""
    return sum(a[..., :, k, None] * b[..., k, None, :] for k in range(3))


def _gell_mann(device):
    s = math.sqrt(3)
    m = torch.zeros(8, 3, 3, dtype=C128)
    m[0, 0, 1] = m[0, 1, 0] = m[3, 0, 2] = m[3, 2, 0] = m[5, 1, 2] = m[5, 2, 1] = 1
    for k, (i, j) in ((1, (0, 1)), (4, (0, 2)), (6, (1, 2))):
        m[k, i, j], m[k, j, i] = -1j, 1j
    m[2, 0, 0], m[2, 1, 1] = 1, -1
    m[7] = torch.diag(torch.tensor([1 / s, 1 / s, -2 / s], dtype=C128))
    return m.to(device)


def _gen(seed, k, device):
    g = torch.Generator(device=device)
    g.manual_seed((int(seed) * 1000003 + k) % (2 ** 62))
    return g


def _gauss(shape, gen, device):
    """Complex Gaussian numbers, Re and Im each N(0, 1), drawn in 32 bits."""
    return torch.view_as_complex(torch.randn(*shape, 2, generator=gen, device=device))


def _links(c, gen, device):
    """SU(3) links exp(i eps H), H = sum_a h_a lambda_a / 2, h_a normal: the recipe of the synthetic fields.

    Taylor series of the quarter angle, squared twice.
    """
    V = math.prod(c["L"])
    h = torch.randn(V * 4, 8, generator=gen, device=device, dtype=torch.float64)
    X = (h.to(C128) @ _gell_mann(device).reshape(8, 9)).reshape(-1, 3, 3) * (0.5j * c["eps"] / 4)
    one = torch.eye(3, dtype=C128, device=device)
    U = one + X / 16
    for k in range(15, 0, -1):
        U = one + _mm3(X, U) / k
    for _ in range(2):
        U = _mm3(U, U)
    return U.reshape(V, 4, 3, 3).contiguous()


def _vector(c, gen, device):
    """Fine right-hand sides in the case's vector type; BF16 as pairs in a last dimension of 2."""
    v = _gauss((math.prod(c["L"]), 4, 3, c["nrhs"]), gen, device)
    if c["prec"] == "bf16":
        return torch.view_as_real(v).to(torch.bfloat16).contiguous()
    return v.to(C128) if c["prec"] == "fp64" else v


def _inputs(c, seed, k, device):
    """Links, test vectors and the right-hand side of lattice k of a case."""
    gen = _gen(seed, k, device)
    U = _links(c, gen, device)
    tv = _gauss((math.prod(c["L"]), 4, 3, c["ntv"]), gen, device).to(C128)
    if c["kind"] == "mixed":  # a coarse right-hand side
        y = _gauss((math.prod(c["L"]) // math.prod(c["B"]), 2, c["ntv"], c["nrhs"]), gen, device)
    else:
        y = None if c["kind"] == "setup" else _vector(c, gen, device)
    return U, tv, y


# ------------------------------------------------------------------ prepare and run
class _Handle:
    """A library handle that is destroyed with its last reference."""

    def __init__(self, params, U, tv):
        self.h, _ = amg.amg_setup_coarse(params, U, tv, torch.cuda.current_stream())

    def __del__(self):
        if getattr(self, "h", None):
            amg.amg_destroy(self.h)


def _params(c, prec=None, max_nrhs=None):
    p = PREC[prec or c["prec"]]
    vec = amg.AMG_FP32 if p == amg.AMG_FP16_SCALED else p
    pair = c.get("arith", "fp64" if c["prec"] == "fp64" else "pair") == "pair"
    return amg.make_params(c["L"], c["B"], c["ntv"], max_nrhs=max_nrhs or c["nrhs"], m0=M0, csw=CSW, link_prec=p,
                           r_prec=vec, vec_prec=vec, setup_arith=amg.AMG_SETUP_F32PAIR if pair else amg.AMG_SETUP_FP64)


def prepare(case, seed):
    state = {"case": case, "kind": case["kind"]}
    handles, ys, xs = [], [], []
    for k, c in enumerate(_parts(case)):
        U, tv, y = _inputs(c, seed, k, "cuda")
        if c["kind"] == "setup":
            Vc, nc = math.prod(c["L"]) // math.prod(c["B"]), 2 * c["ntv"]
            state.update(params=_params(c), U=U, tv=tv,
                         R=torch.empty(Vc, 2, c["ntv"], 6 * math.prod(c["B"]), dtype=C128, device="cuda"),
                         Dc=torch.empty(Vc, 9, nc, nc, dtype=C128, device="cuda"))
            break
        if c["kind"] == "mixed":
            handles.append(_Handle(_params(c, "fp32"), U, tv))
        handles.append(_Handle(_params(c), U, tv))
        if c["kind"] == "cgc_eo":
            amg.amg_setup_evenodd(handles[-1].h, torch.cuda.current_stream())
        if c["kind"] in ("vcycle", "dirac"):
            amg.amg_setup_fine(handles[-1].h, U, torch.cuda.current_stream())
        del U, tv
        ys.append(y)
        xs.append(torch.empty_like(y))
    if case["kind"] == "vcycle":
        state["vp"] = amg.make_vcycle_params(case["tol"], case["restart"], case["max_applies"], case["n_smoother"],
                                             case["n_mr"])
    state.update(handles=handles, y=ys, x=xs)
    torch.cuda.synchronize()  # amg_setup_fine reads U, which goes out of scope here
    return state


def run(state):
    c, kind, st = state["case"], state["kind"], torch.cuda.current_stream()
    if kind == "setup":
        h, _ = amg.amg_setup_coarse(state["params"], state["U"], state["tv"], st)
        amg.amg_export_R(h, state["R"])
        amg.amg_export_Dc(h, state["Dc"])
        amg.amg_destroy(h)
        return state["R"], state["Dc"]
    hs, ys, xs = [h.h for h in state["handles"]], state["y"], state["x"]
    if kind == "batch":
        amg.amg_batch_cgc(hs, ys, xs, [p["nrhs"] for p in _parts(c)], st)
        return xs
    y, x, n = ys[0], xs[0], c["nrhs"]
    if kind == "cgc":
        amg.amg_cgc(hs[0], y, x, n, c["tol"], c["restart"], c["max_applies"], st, info=False)
    elif kind == "cgc_eo":
        amg.amg_cgc_eo(hs[0], y, x, n, c["tol"], c["restart"], c["max_applies"], st, info=False)
    elif kind == "mixed":
        amg.amg_coarse_solve_mixed(hs[0], hs[1], y, x, n, c["tol"], c["inner_tol"], c["restart"], c["max_applies"],
                                   stream=st, info=False)
    elif kind == "vcycle":
        amg.amg_vcycle(hs[0], state["vp"], y, x, n, st)
    else:
        amg.amg_dirac_apply(hs[0], y, x, n, st)
    return x


# ------------------------------------------------------------------ work
def _work_part(c):
    """Bytes and operations of one lattice's pass (a complex multiply-add is 8 operations).

    An input larger than L2 that several dependent steps need (the smoother's links, D_c in a Krylov
    solve) is counted once for each of them.  The coarse solve is counted with two applications of
    D_c, what FGMRES takes to 0.05 on these fields; the mixed solve with three of each operator.
    """
    V, Vb, ntv, r = math.prod(c["L"]), math.prod(c["B"]), c["ntv"], c["nrhs"]
    Vc, nc = V // Vb, 2 * ntv
    z = {"fp64": 16, "fp32": 8, "fp16": 4, "bf16": 4}[c["prec"]]    # bytes of a stored complex number
    zc = 16 if c["prec"] == "fp64" else 8                           # and of a coarse vector's
    nR, nD, nv, ncv = V * 12 * ntv, Vc * 9 * nc * nc, V * 12 * r, Vc * nc * r
    transfer = {"bytes": nR * z + nv * z + ncv * zc, "flops": 8 * nR * r}
    apply = {"bytes": nD * z + 2 * ncv * zc, "flops": 8 * nD * r}
    # D: 8 hops of two 3x3 colour products, projections and sums, two Hermitian 6x6 clover blocks
    dflops = V * r * (8 * (2 * 66 + 36) + 2 * 36 * 8 + 24)
    links, clover = V * 36 * z, V * 42 * z
    kind = c["kind"]
    if kind == "dirac":
        return {"bytes": links + clover + 2 * nv * z, "flops": dflops}
    if kind == "setup":
        # the test vectors' Gram-Schmidt with every projection applied twice, D P and R (D P)
        gs = 2 * 8 * V * 12 * ntv * ntv
        # rank-6 sums: four directions of (2 ntv)^2 entries, the self term's two diagonal quadrants
        asm = 8 * V * 6 * (4 * nc * nc + 2 * ntv * ntv)
        # in: links, test vectors; out: R and D_c in 64 bits and as stored
        return {"bytes": 16 * V * 36 + 2 * 16 * nR + 8 * nR + (16 + 8) * nD, "flops": gs + asm}
    if kind == "batch":
        parts = [transfer, apply, transfer]
    elif kind == "mixed":
        parts = 3 * [apply] + 3 * [{"bytes": nD * 8 + 2 * ncv * 8, "flops": 8 * nD * r}]
    else:
        parts = [transfer, apply, apply, transfer]
    if kind == "vcycle":
        # one half sweep: links, clover, y and x of one colour, x of the other, x written
        half = {"bytes": (links + clover) // 2 + 2 * nv * z, "flops": (1 + c["n_mr"]) * dflops // 2}
        parts += 2 * c["n_smoother"] * [half]
    return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}


def work(case):
    w = [_work_part(c) for c in _parts(case)]
    return {k: sum(p[k] for p in w) for k in ("bytes", "flops")}


# ------------------------------------------------------------------ the method in 64 bits
class _Lattice:
    """D, the aggregates' R, D_c = R D P and the smoother of one lattice, written out in complex128.

    Fine vectors are (t, z, y, x, 4, 3, columns), coarse vectors (Vc, 2, ntv, columns).
    """

    def __init__(self, c, U, tv=None):
        self.c, self.dev = c, U.device
        self.L, self.B = c["L"], c["B"]
        self.shape = tuple(reversed(self.L))
        U = U.reshape(self.shape + (4, 3, 3))
        self.U = [U[..., mu, :, :] for mu in range(4)]
        sig = torch.tensor([[[0, 1], [1, 0]], [[0, -1j], [1j, 0]], [[1, 0], [0, -1]]], dtype=C128)
        self.g = []
        for mu in range(4):
            A = -1j * sig[mu] if mu < 3 else torch.eye(2, dtype=C128)
            G = torch.zeros(4, 4, dtype=C128)
            G[:2, 2:], G[2:, :2] = A, A.conj().T
            self.g.append(G)
        self.clover = self._clover()
        coord = torch.meshgrid(*(torch.arange(n, device=self.dev) for n in self.shape), indexing="ij")
        self.coord = [coord[3 - mu] for mu in range(4)]
        if tv is not None:
            self.Q = self._orthonormal(self._agg(tv.reshape(self.shape + (4, 3, -1))))

    def _shift(self, f, mu, d):
        """f(x + d mu)."""
        return torch.roll(f, -d, 3 - mu)

    def _clover(self):
        out = torch.zeros(self.shape + (4, 3, 4, 3), dtype=C128, device=self.dev)
        dag = lambda m: m.mH
        for mu in range(4):
            for nu in range(mu + 1, 4):
                a, b, s = self.U[mu], self.U[nu], self._shift
                xm, xn = s(a, mu, -1), s(b, nu, -1)                       # U_mu(x-mu), U_nu(x-nu)
                bm, an = s(b, mu, -1), s(a, nu, -1)                       # U_nu(x-mu), U_mu(x-nu)
                q = _mm3(_mm3(a, s(b, mu, 1)), dag(_mm3(b, s(a, nu, 1))))
                q = q + _mm3(_mm3(b, dag(_mm3(bm, s(xm, nu, 1)))), xm)
                q = q + _mm3(dag(_mm3(s(bm, nu, -1), xm)), _mm3(s(xm, nu, -1), xn))
                q = q + _mm3(dag(xn), _mm3(_mm3(an, s(xn, mu, 1)), dag(a)))
                F = (q - dag(q)) / 8
                sig = 0.5j * (self.g[mu] @ self.g[nu] - self.g[nu] @ self.g[mu])
                for i in range(4):
                    for j in range(4):
                        if sig[i, j] != 0:
                            out[..., i, :, j, :] += CSW * 0.5j * complex(sig[i, j]) * F
        return out.reshape(self.shape + (12, 12))

    def _gamma(self, mu, v):
        G, out = self.g[mu], torch.empty_like(v)
        for i in range(4):
            j = int(torch.nonzero(G[i])[0])
            out[..., i, :, :] = complex(G[i, j]) * v[..., j, :, :]
        return out

    def _site(self, v):
        return (4 + M0) * v + (self.clover @ v.reshape(self.shape + (12, -1))).reshape(v.shape)

    def _hop(self, v, mu, d):
        """-1/2 (1 - d gamma_mu) times the link and the neighbour in direction d mu."""
        u = self.U[mu] if d > 0 else self._shift(self.U[mu], mu, -1).mH
        w = torch.zeros_like(v)
        s = self._shift(v, mu, d)
        for k in range(3):
            w += u[..., None, :, k, None] * s[..., :, None, k, :]
        return -0.5 * (w - d * self._gamma(mu, w))

    def _face(self, mu, d):
        """1 where the neighbour in direction d mu lies in another block."""
        m = (self.coord[mu] % self.B[mu]) == (self.B[mu] - 1 if d > 0 else 0)
        return m[..., None, None, None]

    def dirac(self, v, inside=False):
        out = self._site(v)
        for mu in range(4):
            for d in (1, -1):
                h = self._hop(v, mu, d)
                out += h * ~self._face(mu, d) if inside else h
        return out

    # aggregates: (Vc, 2, 6 Vb, columns), dofs (site in block, x fastest; spin of the chirality; colour)
    def _split(self):
        return sum(([self.L[m] // self.B[m], self.B[m]] for m in (3, 2, 1, 0)), [])

    def _agg(self, v):
        k = v.shape[-1]
        v = v.reshape(self._split() + [2, 6, k]).permute(0, 2, 4, 6, 8, 1, 3, 5, 7, 9, 10)
        return v.reshape(-1, 2, 6 * math.prod(self.B), k)

    def _unagg(self, a):
        s, k = self._split(), a.shape[-1]
        a = a.reshape(s[0::2] + [2] + s[1::2] + [6, k]).permute(0, 5, 1, 6, 2, 7, 3, 8, 4, 9, 10)
        return a.reshape(self.shape + (4, 3, k))

    @staticmethod
    def _orthonormal(W):
        """Q of W = Q T with T upper triangular, positive diagonal (Cholesky, applied three times)."""
        for _ in range(3):
            T = torch.linalg.cholesky(W.mH @ W).mH
            W = torch.linalg.solve_triangular(T, W, upper=True, left=False)
        return W

    def restrict(self, v):
        return self.Q.mH @ self._agg(v)

    def prolong(self, xc):
        return self._unagg(self.Q @ xc)

    def coarse(self, xc):
        return self.restrict(self.dirac(self.prolong(xc)))

    def blocks(self, self_only=False):
        """D_c as (Vc, 9, 2 ntv, 2 ntv)."""
        n, Vc = self.Q.shape[-1], self.Q.shape[0]
        out = torch.zeros(Vc, 1 if self_only else 9, 2 * n, 2 * n, dtype=C128, device=self.dev)
        for hc in range(2):
            Q = self.Q.clone()
            Q[:, 1 - hc] = 0
            v = self._unagg(Q)
            cols = slice(hc * n, hc * n + n)
            out[:, 0, :, cols] = self.restrict(self.dirac(v, inside=True)).reshape(Vc, 2 * n, n)
            for mu in range(0 if self_only else 4):
                for k, d in ((1, 1), (2, -1)):
                    w = self._hop(v, mu, d) * self._face(mu, d)
                    out[:, 2 * mu + k, :, cols] = self.restrict(w).reshape(Vc, 2 * n, n)
        return out

    def sap(self, y, x, cycles, n_mr):
        """Alg. 3: multiplicative Schwarz over two block colours, n_mr minimal-residual steps per block."""
        colour = sum(self.coord[mu] // self.B[mu] for mu in range(4)) % 2
        Vc = math.prod(self.L) // math.prod(self.B)

        def dot(a, b):  # per block and column, spread over the block's sites
            s = self._agg(a.conj() * b).sum((1, 2), keepdim=True)
            return self._unagg(s.expand(Vc, 2, 6 * math.prod(self.B), s.shape[-1]))

        for _ in range(cycles):
            for c in range(2):
                on = (colour == c)[..., None, None, None]
                rho = (y - self.dirac(x)) * on
                e = torch.zeros_like(x)
                for _ in range(n_mr):
                    p = self.dirac(rho, inside=True)
                    den = dot(p, p)
                    al = torch.where(den == 0, 0, dot(p, rho) / torch.where(den == 0, 1, den))
                    e = e + al * rho
                    rho = rho - al * p
                x = x + e
        return x


def _gmres(A, b, tol, m, max_applies):
    """First cycle of GMRES(m) from zero, every column on its own; None when a column needs more."""
    shape, r = b.shape, b.shape[-1]
    b = b.reshape(-1, r)
    beta = torch.linalg.vector_norm(b, dim=0)
    V = [b / beta]
    H = torch.zeros(r, m + 1, m, dtype=C128)
    x = torch.zeros_like(b)
    left = set(range(r))
    for j in range(min(m, max_applies)):
        w = A(V[j].reshape(shape)).reshape(-1, r)
        for _ in range(2):
            h = torch.stack([(v.conj() * w).sum(0) for v in V])
            w = w - sum(h[i] * V[i] for i in range(j + 1))
            H[:, :j + 1, j] += h.T.cpu()
        n = torch.linalg.vector_norm(w, dim=0)
        H[:, j + 1, j] = n.cpu()
        V.append(w / n)
        for k in sorted(left):
            rhs = torch.zeros(j + 2, 1, dtype=C128)
            rhs[0] = beta[k].cpu()
            Hk = H[k, :j + 2, :j + 1]
            yk = torch.linalg.lstsq(Hk, rhs).solution
            if torch.linalg.vector_norm(rhs - Hk @ yk) <= tol * beta[k].cpu():
                x[:, k] = sum(complex(yk[i, 0]) * V[i][:, k] for i in range(j + 1))
                left.discard(k)
        if not left:
            return x.reshape(shape)
    return None


def _coarse_solve(lat, c, b):
    if c["kind"] != "cgc_eo":
        return _gmres(lat.coarse, b, c["tol"], c["restart"], c["max_applies"])
    # Schur complement on the even sites; half vectors kept full with zeros on the other parity
    Lc = [n // m for n, m in zip(lat.L, lat.B)]
    i = torch.arange(math.prod(Lc), device=b.device)
    par = (i % Lc[0] + i // Lc[0] % Lc[1] + i // (Lc[0] * Lc[1]) % Lc[2] + i // (Lc[0] * Lc[1] * Lc[2])) % 2
    even = (par == 0).reshape(-1, 1, 1, 1)
    S = lat.blocks(self_only=True)[:, 0]
    mul = lambda M, v: (M @ v.reshape(v.shape[0], -1, v.shape[-1])).reshape(v.shape)
    Sinv = torch.linalg.inv(S)
    hop = lambda v: lat.coarse(v) - mul(S, v)
    schur = lambda v: mul(S, v) - hop(mul(Sinv, hop(v) * ~even)) * even
    xe = _gmres(schur, b * even - hop(mul(Sinv, b * ~even)) * even, c["tol"], c["restart"], c["max_applies"])
    return None if xe is None else xe + mul(Sinv, (b - hop(xe)) * ~even)


def _exact_part(c, seed, k, device):
    U, tv, y = _inputs(c, seed, k, device)
    lat = _Lattice(c, U, None if c["kind"] == "dirac" else tv)
    del U, tv
    if c["kind"] == "setup":
        return lat.Q.mH.resolve_conj().contiguous(), lat.blocks()
    v = torch.view_as_complex(y.double()) if c["prec"] == "bf16" else y.to(C128)
    v = v.reshape(lat.shape + v.shape[1:])
    if c["kind"] == "dirac":
        x = lat.dirac(v)
    elif c["kind"] == "batch":
        x = lat.prolong(lat.coarse(lat.restrict(v)))
    else:
        xc = _coarse_solve(lat, c, lat.restrict(v))
        if xc is None:
            return None
        x = lat.prolong(xc)
        if c["kind"] == "vcycle":
            x = lat.sap(v, x, c["n_smoother"], c["n_mr"])
    x = x.reshape(math.prod(c["L"]), 4, 3, -1)
    return torch.view_as_real(x).contiguous() if c["prec"] == "bf16" else x


def exact(case, seed, device="cuda"):
    """None for the mixed solve: any vector with a true residual below its tolerance is a result."""
    if case["kind"] == "mixed":
        return None
    out = [_exact_part(c, seed, k, device) for k, c in enumerate(_parts(case))]
    return out if case["kind"] == "batch" else out[0]
