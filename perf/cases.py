"""The work a user of this library has it do, as measurable cases.

Every case goes through the public Python calls (fsgpu, autograd).  The listed
cases span the real range of the library: from one gate on a 4900-amplitude
state, where launches and host work count, to a forward pass and its gradient
on 1.66e8 amplitudes; both precisions; closed and open, square and ragged
sectors; single circuits, a batch, a Trotter evolution, a Hamiltonian action
and sampling.  `draw` gives further cases of the same ranges.
"""

import math

import numpy as np
import torch

DEVICE = "cuda" if torch.cuda.is_available() else "cpu"


def listed():
    return [
        # one gate layer on the smallest documented state, the way a script
        # or an interactive session applies gates one by one
        dict(name="gates_small_c128", kind="gates", norb=8, na=4, nb=4, dtype="c128", spinful=False),
        # an open-shell sector with its own matrices per spin and odd
        # dimensions (1287 x 1716)
        dict(name="gates_ragged_c64", kind="gates", norb=13, na=5, nb=7, dtype="c64", spinful=True),
        # the plain method on a mid-size state in the default precision
        dict(name="gates_mid_c128", kind="gates", norb=14, na=7, nb=7, dtype="c128", spinful=False),
        # the plain method at scale
        dict(name="gates_large_c64", kind="gates", norb=16, na=8, nb=8, dtype="c64", spinful=False),
        # one optimisation step of a small ansatz (value and gradient), in
        # both precisions
        dict(name="lucj_small_c64", kind="lucj", norb=12, na=6, nb=6, dtype="c64", reps=4,
             from_hf=True),
        dict(name="lucj_small_c128", kind="lucj", norb=12, na=6, nb=6, dtype="c128", reps=4,
             from_hf=True),
        # an optimisation step on the headline state (two repetitions)
        dict(name="lucj_large_c64", kind="lucj", norb=16, na=8, nb=8, dtype="c64", reps=2,
             from_hf=False),
        # many small uneven circuits at once: a parameter sweep
        dict(name="batch_c64", kind="batch", circuits=24, dtype="c64", reps=2),
        # time evolution by a double-factorized Hamiltonian, open shell
        dict(name="trotter_c128", kind="trotter", norb=11, na=6, nb=5, dtype="c128", terms=3,
             steps=3, order=0),
        # one Hamiltonian action of an eigensolver, in both precisions
        dict(name="operator_c64", kind="operator", norb=12, na=6, nb=6, dtype="c64"),
        dict(name="operator_c128", kind="operator", norb=10, na=5, nb=5, dtype="c128"),
        # measurement shots from a large state
        dict(name="sample_c64", kind="sample", norb=15, na=7, nb=8, dtype="c64", shots=1000000),
    ]


def _amplitudes(c):
    return math.comb(c["norb"], c["na"]) * math.comb(c["norb"], c["nb"])


def _sector(rng, lo, hi, most, least=1):
    """A sector of lo .. hi orbitals around half filling with at most `most`
    (and at least `least`) amplitudes."""
    while True:
        norb = rng.randint(lo, hi)
        na = min(norb - 1, max(1, norb // 2 + rng.randint(-3, 1)))
        nb = min(norb - 1, max(1, norb // 2 + rng.randint(-3, 1)))
        s = dict(norb=norb, na=na, nb=nb)
        if least <= _amplitudes(s) <= most:
            return s


def draw(rng):
    kind = rng.choice(["gates", "gates", "gates", "lucj", "lucj", "lucj", "batch", "trotter",
                       "trotter", "operator", "sample"])
    dtype = rng.choice(["c64", "c128"])
    c64 = dtype == "c64"
    if kind == "gates":
        s = _sector(rng, 8, 16, 170e6 if c64 else 42e6)
        return dict(kind=kind, dtype=dtype, spinful=rng.random() < 0.5, **s)
    if kind == "lucj":
        s = _sector(rng, 8, 15 if c64 else 13, 42e6 if c64 else 3e6)
        return dict(kind=kind, dtype=dtype, reps=rng.randint(1, 4 if _amplitudes(s) < 12e6 else 2),
                    from_hf=rng.random() < 0.5, **s)
    if kind == "batch":
        return dict(kind=kind, dtype="c64", circuits=rng.randint(4, 24), reps=rng.randint(1, 2))
    if kind == "trotter":
        s = _sector(rng, 8, 15 if c64 else 13, 42e6 if c64 else 3e6)
        big = _amplitudes(s) > 12e6
        return dict(kind=kind, dtype=dtype, terms=rng.randint(1, 2 if big else 4),
                    steps=rng.randint(1, 2 if big else 3), order=0 if big else rng.randint(0, 1), **s)
    if kind == "operator":
        s = _sector(rng, 8, 12, 860e3 if c64 else 64e3, 1000)
        return dict(kind=kind, dtype=dtype, **s)
    s = _sector(rng, 8, 15, 42e6, 1000)
    return dict(kind=kind, dtype=dtype, shots=int(10 ** rng.uniform(3, 6)), **s)


# ------------------------------------------------------------------ inputs
def _haar(n, g):
    z = g.standard_normal((n, n)) + 1j * g.standard_normal((n, n))
    q, r = np.linalg.qr(z)
    d = np.diag(r)
    return q * (d / np.abs(d))[None, :]


def _symmetric(n, sigma, g):
    a = np.triu(g.normal(0.0, sigma, (n, n)))
    return a + np.triu(a, 1).T


def _antihermitian(n, sigma, g):
    up = np.triu(g.normal(0.0, sigma, (n, n)) + 1j * g.normal(0.0, sigma, (n, n)), 1)
    return up - up.conj().T + np.diag(1j * g.normal(0.0, sigma, n))


def _log_haar(n, g):
    """An anti-Hermitian generator of a dense random rotation: a random basis
    with angles spread over (-pi, pi)."""
    z = _haar(n, g)
    k = (z * (1j * g.uniform(-math.pi, math.pi, n))[None, :]) @ z.conj().T
    return 0.5 * (k - k.conj().T)


def _line_couplings(n, sigma, g):
    """J_aa on nearest neighbours of a line, J_ab on the same site."""
    jaa = np.diag(g.normal(0.0, sigma, n - 1), 1)
    return jaa + jaa.T, np.diag(g.normal(0.0, sigma, n))


def _state(norb, na, nb, dtype, seed):
    """A normalised random state drawn on the device."""
    gen = torch.Generator(device=DEVICE)
    gen.manual_seed(int(seed))
    real = torch.float32 if dtype == "c64" else torch.float64
    v = torch.randn((math.comb(norb, na), math.comb(norb, nb), 2), generator=gen, device=DEVICE,
                    dtype=real)
    v = torch.view_as_complex(v)
    return v / torch.linalg.vector_norm(v)


def _lucj_params(norb, reps, small, g):
    K, Ja, Jb = [], [], []
    for _ in range(reps):
        if small:  # starting point of an optimisation: weak rotations, local couplings
            K.append(_antihermitian(norb, 0.1, g))
            a, b = _line_couplings(norb, 0.1, g)
        else:  # dense rotations and couplings
            K.append(_log_haar(norb, g))
            a, b = 0.3 * _symmetric(norb, 0.5, g), 0.3 * _symmetric(norb, 0.5, g)
        Ja.append(a)
        Jb.append(b)
    return np.array(K), np.array(Ja), np.array(Jb)


_BATCH_NORBS = (8, 10, 12, 14)


def prepare(case, seed):
    c = dict(case)
    g = np.random.Generator(np.random.PCG64(seed))
    kind = c["kind"]
    if kind == "batch":
        circuits, vecs, cots = [], [], []
        for i in range(c["circuits"]):
            n = _BATCH_NORBS[i % len(_BATCH_NORBS)]
            K, Ja, Jb = _lucj_params(n, c["reps"], False, g)
            circuits.append(dict(K=K, J_aa=Ja, J_ab=Jb, norb=n, nelec=(n // 2, n // 2),
                                 from_hf=True))
            cots.append(_state(n, n // 2, n // 2, c["dtype"], seed * 64 + i))
            vecs.append(torch.empty_like(cots[-1]))
        return dict(case=c, circuits=circuits, vecs=vecs, cots=cots)
    n = c["norb"]
    s = dict(case=c, norb=n, nelec=(c["na"], c["nb"]))
    s["vec"] = _state(n, c["na"], c["nb"], c["dtype"], 2 * seed)
    if kind == "gates":
        s["U"] = _haar(n, g)
        s["U_b"] = _haar(n, g) if c["spinful"] else None
        s["J_aa"], s["J_ab"] = _symmetric(n, 0.5, g), _symmetric(n, 0.5, g)
        s["J_bb"] = _symmetric(n, 0.5, g) if c["spinful"] else None
        s["t"] = 0.3
    elif kind == "lucj":
        K, Ja, Jb = _lucj_params(n, c["reps"], c["from_hf"], g)
        s["K"] = torch.from_numpy(K).requires_grad_(True)
        s["J_aa"] = torch.from_numpy(Ja).requires_grad_(True)
        s["J_ab"] = torch.from_numpy(Jb).requires_grad_(True)
        s["cot"] = _state(n, c["na"], c["nb"], c["dtype"], 2 * seed + 1)
        if not c["from_hf"]:
            s["vec"].requires_grad_(True)
    elif kind == "trotter":
        a = g.normal(0, 0.5, (n, n)) + 1j * g.normal(0, 0.5, (n, n))
        s["h"] = (a + a.conj().T) / 2
        s["J"] = np.array([_symmetric(n, 0.5, g) for _ in range(c["terms"])])
        s["U"] = np.array([_haar(n, g) for _ in range(c["terms"])])
        s["time"] = 1.0
    elif kind == "operator":
        a, b = g.normal(0, 1, (n, n)), g.normal(0, 0.5, (n, n, n, n))
        s["h1"] = (a + a.T) / 2
        s["h2"] = (b + b.transpose(1, 0, 3, 2) + b.transpose(2, 3, 0, 1) + b.transpose(3, 2, 1, 0)) / 4
        s["constant"] = 0.7
    elif kind == "sample":
        gen = torch.Generator(device=DEVICE)
        gen.manual_seed(seed)
        s["uniforms"] = torch.rand(c["shots"], dtype=torch.float64, device=DEVICE, generator=gen)
    else:
        raise ValueError(kind)
    return s


# --------------------------------------------------------------------- run
def run(s):
    from paper_2605_03123_gb300 import autograd, fsgpu
    kind = s["case"]["kind"]
    if kind == "batch":
        grads = fsgpu.lucj_batch_(s["vecs"], s["cots"], s["circuits"])
        flat = [np.concatenate([x[k].ravel() for x in grads]) for k in range(3)]
        return dict(inputs=s["vecs"], cots=s["cots"], dK=flat[0], dJ_aa=flat[1], dJ_ab=flat[2])
    n, ne = s["norb"], s["nelec"]
    if kind == "gates":
        x = fsgpu.apply_orbital_rotation(s["vec"], s["U"], n, ne, U_b=s["U_b"])
        return fsgpu.apply_diag_coulomb_evolution_(x, s["J_aa"], s["J_ab"], s["t"], n, ne,
                                                   J_bb=s["J_bb"])
    if kind == "lucj":
        hf = s["case"]["from_hf"]
        out = autograd.lucj(s["vec"], s["K"], s["J_aa"], s["J_ab"], n, ne, from_hf=hf)
        wrt = [s["K"], s["J_aa"], s["J_ab"]] + ([] if hf else [s["vec"]])
        grads = torch.autograd.grad(out, wrt, grad_outputs=s["cot"])
        return dict(out=out.detach(), grads=list(grads))
    if kind == "trotter":
        x = s["vec"].clone()
        c = s["case"]
        return fsgpu.simulate_trotter_double_factorized_(x, s["h"], s["J"], s["U"], s["time"], n,
                                                         ne, n_steps=c["steps"], order=c["order"])
    if kind == "operator":
        return fsgpu.apply_molecular_hamiltonian(s["vec"], s["h1"], s["h2"], n, ne,
                                                 constant=s["constant"])
    return fsgpu.sample_state(s["vec"], n, ne, uniforms=s["uniforms"])


# -------------------------------------------------------------------- work
def _rotation_flops(norb, na, nb):
    """Real flops per amplitude of one orbital rotation of both spins: 10 per
    amplitude and Givens rotation that moves it, N(N-1)/2 rotations a spin,
    each moving 2 C(N-2, n-1) of the C(N, n) strings."""
    return sum(10 * norb * (norb - 1) / 2 * 2 * math.comb(norb - 2, k - 1) / math.comb(norb, k)
               for k in (na, nb) if 0 < k < norb)


def work(case):
    c = case
    size = 8 if c["dtype"] == "c64" else 16
    if c["kind"] == "batch":
        by = fl = 0.0
        for i in range(c["circuits"]):
            n = _BATCH_NORBS[i % len(_BATCH_NORBS)]
            w = work(dict(kind="lucj", norb=n, na=n // 2, nb=n // 2, dtype=c["dtype"],
                          reps=c["reps"], from_hf=True))
            by += w["bytes"]
            fl += w["flops"]
        return dict(bytes=by, flops=fl)
    n, na, nb = c["norb"], c["na"], c["nb"]
    amps = _amplitudes(c)
    rot = _rotation_flops(n, na, nb)
    if c["kind"] == "gates":
        return dict(bytes=2.0 * size * amps, flops=amps * (rot + 12.0))
    if c["kind"] == "lucj":
        # forward, then both states backwards with the transition sums
        # (8 flops per amplitude and single excitation) and the coupling sums
        nrot = c["reps"] + 1
        fwd = (nrot - (1 if c["from_hf"] else 0)) * rot + c["reps"] * 12.0
        rev = nrot * (2 * rot + 8.0 * (na * (n - na + 1) + nb * (n - nb + 1))) + c["reps"] * 30.0
        states = 2.0 + (0.0 if c["from_hf"] else 2.0)  # out, cot (, vec, its gradient)
        return dict(bytes=states * size * amps, flops=amps * (fwd + rev))
    if c["kind"] == "trotter":
        # one rotation and one evolution per two-body term and stage
        stages = c["steps"] * (1 if c["order"] == 0 else 2)
        return dict(bytes=2.0 * size * amps,
                    flops=amps * (stages * c["terms"] * (rot + 12.0) + rot))
    if c["kind"] == "operator":
        # two contractions of the N^2 x N^2 tensor (same spin, mixed) over
        # the nonzero excitations of each amplitude, and the outer sums
        ex = na * (n - na + 1) + nb * (n - nb + 1)
        return dict(bytes=2.0 * size * amps, flops=amps * (4.0 * n * n * ex + 4.0 * ex))
    return dict(bytes=1.0 * size * amps + 16.0 * c["shots"], flops=4.0 * amps)


# ------------------------------------------------------------ 64-bit values
# Plain torch in complex128, from the definitions: adjacent Givens rotations
# on lists of strings, phases per configuration, dense single excitations.
class _Strings:
    def __init__(self, norb, nocc):
        self.norb = norb
        m = [x for x in range(1 << norb) if bin(x).count("1") == nocc]
        self.masks = np.array(m, dtype=np.int64)
        self.index = np.full(1 << norb, -1, dtype=np.int64)
        self.index[self.masks] = np.arange(len(m))
        self.occ = torch.from_numpy(((self.masks[:, None] >> np.arange(norb)) & 1)
                                    .astype(np.float64)).to(DEVICE)
        self._ex = {}

    def excite(self, p, q):
        """(source, target, sign) of a^dag_p a_q over the strings."""
        if (p, q) not in self._ex:
            m = self.masks
            ok = ((m >> q) & 1 == 1) & ((p == q) | ((m >> p) & 1 == 0))
            src = np.nonzero(ok)[0]
            s = m[src]
            t = (s ^ (1 << q)) | (1 << p)
            lo, hi = min(p, q), max(p, q)
            between = s & (((1 << hi) - 1) & ~((2 << lo) - 1)) if p != q else 0 * s
            sg = np.ones(len(src))
            for k in range(self.norb):
                sg *= 1.0 - 2.0 * ((between >> k) & 1)
            self._ex[p, q] = (torch.from_numpy(src).to(DEVICE),
                              torch.from_numpy(self.index[t]).to(DEVICE),
                              torch.from_numpy(sg).to(DEVICE))
        return self._ex[p, q]


def _rotate_rows(v, U, st):
    """v[i, :] over the strings of one spin -> the orbital rotation by U."""
    n = st.norb
    A = np.array(U, dtype=np.complex128)
    gs = []
    for j in range(n):
        for q in range(n - 1, j, -1):
            a, b = A[q - 1, j], A[q, j]
            r = math.hypot(abs(a), abs(b))
            if abs(b) == 0.0:
                continue
            G = np.array([[a.conjugate() / r, b.conjugate() / r], [-b / r, a / r]])
            A[q - 1:q + 1] = G @ A[q - 1:q + 1]
            gs.append((q - 1, a / r, b / r))
    ph = torch.from_numpy(np.angle(np.diag(A))).to(DEVICE)
    ang = st.occ @ ph
    v = v * torch.polar(torch.ones_like(ang), ang)[:, None]
    for p, a, b in reversed(gs):
        dst, src, _ = st.excite(p, p + 1)  # dst: p + 1 occupied, src: p occupied
        x, y = v.index_select(0, src), v.index_select(0, dst)
        v.index_copy_(0, src, complex(a) * x - complex(b.conjugate()) * y)
        v.index_copy_(0, dst, complex(b) * x + complex(a.conjugate()) * y)
    return v


def _rotate(v, Ua, Ub, sa, sb):
    v = _rotate_rows(v, Ua, sa)
    return _rotate_rows(v.t().contiguous(), Ub, sb).t().contiguous()


def _coulomb(v, Jaa, Jab, Jbb, t, sa, sb):
    dev = lambda x: torch.from_numpy(np.ascontiguousarray(x, dtype=np.float64)).to(DEVICE)
    qa = torch.einsum("ip,pq,iq->i", sa.occ, dev(Jaa), sa.occ)
    qb = torch.einsum("ip,pq,iq->i", sb.occ, dev(Jbb), sb.occ)
    x = sa.occ @ dev(Jab)
    out = torch.empty_like(v)
    for i in range(0, v.shape[0], 1024):
        ang = -0.5 * t * (qa[i:i + 1024, None] + qb[None, :] + 2.0 * (x[i:i + 1024] @ sb.occ.t()))
        out[i:i + 1024] = v[i:i + 1024] * torch.polar(torch.ones_like(ang), ang)
    return out


def _transitions(psi, g, sa, sb):
    """T[p, q] = <g| sum over spins of a^dag_p a_q |psi>."""
    n = sa.norb
    T = np.zeros((n, n), dtype=np.complex128)
    for st, flip in ((sa, False), (sb, True)):
        if len(st.masks) == 0:
            continue
        P, G = (psi.t().contiguous(), g.t().contiguous()) if flip else (psi, g)
        acc = torch.zeros((n, n), dtype=torch.complex128, device=DEVICE)
        for p in range(n):
            for q in range(n):
                src, dst, sg = st.excite(p, q)
                for i in range(0, len(src), 4096):
                    x = P.index_select(0, src[i:i + 4096])
                    x *= sg[i:i + 4096, None]
                    acc[p, q] += torch.vdot(G.index_select(0, dst[i:i + 4096]).view(-1), x.view(-1))
        T += acc.cpu().numpy()
    return T


def _expm(K):
    return torch.matrix_exp(torch.from_numpy(np.ascontiguousarray(K))).numpy()


def _lucj_exact(vec, cot, K, Ja, Jb, sa, sb, from_hf):
    """(out, dK, dJ_aa, dJ_ab, d vec) of the ansatz and its gradient."""
    reps = K.shape[0]
    psi = vec
    if from_hf:
        psi = torch.zeros((len(sa.masks), len(sb.masks)), dtype=torch.complex128, device=DEVICE)
        psi[0, 0] = 1.0
    Us = [_expm(K[k]) for k in range(reps)]
    for k in range(reps):
        psi = _rotate(psi.clone(), Us[k].conj().T, Us[k].conj().T, sa, sb)
        psi = _coulomb(psi, Ja[k], Jb[k], Ja[k], 1.0, sa, sb)
        psi = _rotate(psi, Us[k], Us[k], sa, sb)
    out, g = psi, cot
    dK, dJa, dJb = np.zeros_like(K), np.zeros_like(Ja), np.zeros_like(Jb)
    for k in reversed(range(reps)):
        Ud = Us[k].conj().T
        T1 = _transitions(psi, g, sa, sb)
        psi, g = _rotate(psi.clone(), Ud, Ud, sa, sb), _rotate(g.clone(), Ud, Ud, sa, sb)
        W = (g.conj() * psi).imag
        dJb[k] = (sa.occ.t() @ W @ sb.occ).cpu().numpy()
        wa, wb = W.sum(1), W.sum(0)
        dJa[k] = 0.5 * (sa.occ.t() @ (wa[:, None] * sa.occ)
                        + sb.occ.t() @ (wb[:, None] * sb.occ)).cpu().numpy()
        del W
        psi = _coulomb(psi, Ja[k], Jb[k], Ja[k], -1.0, sa, sb)
        g = _coulomb(g, Ja[k], Jb[k], Ja[k], -1.0, sa, sb)
        T2 = _transitions(psi, g, sa, sb)
        psi, g = _rotate(psi, Us[k], Us[k], sa, sb), _rotate(g, Us[k], Us[k], sa, sb)
        # d Re<g|psi> = Re sum_pq (dU U^dag)_pq T_pq at each rotation
        Kt = torch.from_numpy(K[k].copy()).requires_grad_(True)
        E = torch.matrix_exp(Kt)
        U0 = torch.from_numpy(Us[k])
        f = ((E @ U0.conj().t()) * torch.from_numpy(T1)).sum().real
        f = f + ((E.conj().t() @ U0) * torch.from_numpy(T2)).sum().real
        f.backward()
        dK[k] = Kt.grad.numpy()
    return out, dK, dJa, dJb, g


def _operator_exact(v, h1, h2, constant, sa, sb):
    n = sa.norb
    da, db = v.shape
    one = torch.from_numpy(h1 - 0.5 * np.einsum("prrq->pq", h2)).to(DEVICE)
    two = torch.from_numpy(h2.reshape(n * n, n * n)).to(DEVICE)

    def excited(x, p, q):
        out = torch.zeros_like(x)
        src, dst, sg = sa.excite(p, q)
        out.index_add_(0, dst, x.index_select(0, src) * sg[:, None])
        src, dst, sg = sb.excite(p, q)
        out.index_add_(1, dst, x.index_select(1, src) * sg[None, :])
        return out

    D = torch.stack([excited(v, p, q).view(-1) for p in range(n) for q in range(n)])
    Dr = torch.view_as_real(D).reshape(n * n, -1)
    one_v = constant * v + torch.view_as_complex(
        (one.reshape(1, -1) @ Dr).reshape(da, db, 2).contiguous())
    G = 0.5 * (two @ Dr)
    del D, Dr
    for p in range(n):
        for q in range(n):
            one_v += excited(torch.view_as_complex(G[p * n + q].reshape(da, db, 2)), p, q)
    return one_v


def exact(case, seed):
    c = case
    if c["kind"] == "sample":
        return None
    s = prepare(case, seed)
    with torch.no_grad():
        if c["kind"] == "batch":
            ins, cots, dK, dJa, dJb = [], [], [], [], []
            tables = {n: _Strings(n, n // 2) for n in _BATCH_NORBS}
            for cir, cot in zip(s["circuits"], s["cots"]):
                st = tables[cir["norb"]]
                with torch.enable_grad():
                    _, a, b, d, g = _lucj_exact(None, cot.to(torch.complex128), cir["K"],
                                                cir["J_aa"], cir["J_ab"], st, st, True)
                hf = torch.zeros_like(g)
                hf[0, 0] = 1.0
                ins.append(hf)
                cots.append(g)
                dK.append(a.ravel())
                dJa.append(b.ravel())
                dJb.append(d.ravel())
            return dict(inputs=ins, cots=cots, dK=np.concatenate(dK), dJ_aa=np.concatenate(dJa),
                        dJ_ab=np.concatenate(dJb))
        n = c["norb"]
        sa, sb = _Strings(n, c["na"]), _Strings(n, c["nb"])
        v = s["vec"].detach().to(torch.complex128)
        if c["kind"] == "gates":
            U_b = s["U"] if s["U_b"] is None else s["U_b"]
            J_bb = s["J_aa"] if s["J_bb"] is None else s["J_bb"]
            return _coulomb(_rotate(v.clone(), s["U"], U_b, sa, sb), s["J_aa"], s["J_ab"], J_bb,
                            s["t"], sa, sb)
        if c["kind"] == "lucj":
            with torch.enable_grad():
                out, dK, dJa, dJb, g = _lucj_exact(
                    v, s["cot"].to(torch.complex128), s["K"].detach().numpy(),
                    s["J_aa"].detach().numpy(), s["J_ab"].detach().numpy(), sa, sb, c["from_hf"])
            return dict(out=out, grads=[dK, dJa, dJb] + ([] if c["from_hf"] else [g]))
        if c["kind"] == "trotter":
            dt = s["time"] / c["steps"]
            terms = list(range(c["terms"] + 1))
            seq = [(k, dt) for k in terms] if c["order"] == 0 else \
                [(k, dt / 2) for k in terms] + [(k, dt / 2) for k in reversed(terms)]
            for _ in range(c["steps"]):
                for k, t in seq:
                    if k == 0:
                        E = _expm(-1j * t * s["h"])
                        v = _rotate(v.clone(), E, E, sa, sb)
                        continue
                    U, J = s["U"][k - 1], s["J"][k - 1]
                    v = _rotate(v.clone(), U.conj().T, U.conj().T, sa, sb)
                    v = _coulomb(v, J, J, J, t, sa, sb)
                    v = _rotate(v, U, U, sa, sb)
            return v
        return _operator_exact(v, s["h1"], s["h2"], s["constant"], sa, sb)
