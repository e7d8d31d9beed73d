"""Cases that stand for what a program does with this library, each run through its public entry points.

A case is one of four kinds of call:
  solve    the structure is on the device already (a context per structure); one pass solves its columns,
           takes the density and energy-density matrices on the device and the energies.  A program that
           moves atoms or scans temperatures and electron counts spends its time here.
  request  the whole calculation from host arrays to host arrays: setup, solve, density, energy, destroy.
  serve    several requests at once through the request server, densities returned to the host.
  outputs  what is asked of a solved context: atomic forces and G(z) on a list of shifts.
Structures are those of the repository's generators: jittered diamond, random-packed amorphous carbon and
fluorene-like polymer chains (hydrogens with padding orbitals).  A case fixes the structure and its neighbour
list; the seed moves the matrix elements on it, as a step of a molecular-dynamics run with a kept neighbour
list or of a self-consistent potential does.
"""

import math

import numpy as np
import torch

import paper_1307_3218_gb300 as m
import tbsynth

PRECISION = {"fp64": m.MARNOLDI_FP64, "mixed": m.MARNOLDI_MIXED}


def listed():
    return [
        # the smallest whole calculation: one 64-atom cell, kept on the device; launches and host work count
        {"name": "cell64-fp64", "kind": "solve", "structure": "diamond", "size": 2, "precision": "fp64",
         "nu": 30, "region": 0, "share": 1, "kT": 0.1},
        # the same cell as a new request each time: validation, upload, solve, read-back
        {"name": "cell64-request", "kind": "request", "structure": "diamond", "size": 2, "precision": "mixed",
         "nu": 30, "region": 0, "share": 1, "kT": 0.1},
        # a queue of small amorphous structures of several sizes through the request server
        {"name": "serve-small", "kind": "serve", "structure": "amorphous", "size": 100, "requests": 16,
         "precision": "mixed", "nu": 30, "region": 0, "share": 1, "kT": 0.1},
        # an ordinary structure in each precision; atoms not a multiple of the tile of 8
        {"name": "amorphous1001-fp64", "kind": "solve", "structure": "amorphous", "size": 1001, "precision": "fp64",
         "nu": 30, "region": 0, "share": 1, "kT": 0.1},
        {"name": "amorphous2048-mixed", "kind": "solve", "structure": "amorphous", "size": 2048,
         "precision": "mixed", "nu": 30, "region": 0, "share": 1, "kT": 0.1},
        # larger subspaces (nu typically 30 to 300), on a structure of the serving trace
        {"name": "amorphous512-nu100", "kind": "solve", "structure": "amorphous", "size": 512, "precision": "mixed",
         "nu": 100, "region": 0, "share": 1, "kT": 0.1},
        # the benchmark structure, every column
        {"name": "amorphous4096-mixed", "kind": "solve", "structure": "amorphous", "size": 4096,
         "precision": "mixed", "nu": 30, "region": 0, "share": 1, "kT": 0.1},
        # one rank's share of its columns (an eighth) in FP64 at the shared Fermi level
        {"name": "amorphous4096-fp64-share", "kind": "solve", "structure": "amorphous", "size": 4096,
         "precision": "fp64", "nu": 30, "region": 0, "share": 8, "kT": 0.1},
        # a structure beyond global mode: 256-atom regions, every column
        {"name": "regional6000-mixed", "kind": "solve", "structure": "amorphous", "size": 6000,
         "precision": "mixed", "nu": 30, "region": 256, "share": 1, "kT": 0.1},
        # one rank's share of such a structure at nu = 100
        {"name": "regional6000-nu100-share", "kind": "solve", "structure": "amorphous", "size": 6000,
         "precision": "mixed", "nu": 100, "region": 256, "share": 6, "kT": 0.1},
        # a polymer chain with the largest usual subspace, a share of its columns
        {"name": "polymer12-nu300-share", "kind": "solve", "structure": "polymer", "size": 12, "precision": "fp64",
         "nu": 300, "region": 0, "share": 6, "kT": 0.1},
        # forces and the Green's function on a contour, from a solved context
        {"name": "forces-green", "kind": "outputs", "structure": "amorphous", "size": 1001, "precision": "mixed",
         "nu": 30, "region": 0, "share": 1, "kT": 0.1, "shifts": 8},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "solve", "request", "serve", "outputs"])
    case = {"kind": kind, "precision": rng.choice(["fp64", "mixed", "mixed"]), "region": 0, "share": 1,
            "kT": rng.choice([0.05, 0.1, 0.2])}
    if kind == "serve":
        case.update(structure=rng.choice(["amorphous", "polymer"]), requests=rng.randint(2, 24), nu=rng.randint(12, 40))
        case["size"] = _log_int(rng, 64, 400) if case["structure"] == "amorphous" else rng.randint(2, 4)
        return case
    if kind == "solve" and rng.random() < 0.3:   # regional
        case.update(structure="amorphous", size=_log_int(rng, 2000, 8000), region=rng.choice([100, 192, 256, 300]),
                    nu=_log_int(rng, 20, 100))
    else:
        case["structure"] = rng.choice(["diamond", "amorphous", "amorphous", "polymer"])
        if case["structure"] == "diamond":
            case["size"] = rng.randint(2, 5)
        elif case["structure"] == "polymer":
            case["size"] = rng.randint(4, 24)
        else:
            case["size"] = _log_int(rng, 100, 4096 if kind == "solve" else 1500)
        case["nu"] = _log_int(rng, 12, 250 if kind == "solve" else 60)
        if kind == "outputs":
            case["shifts"] = rng.randint(1, 16)
    atoms = _atoms(case)
    case["nu"] = min(case["nu"], atoms)   # well below the dense limit, as the method is used
    # keep the pass within the largest listed one: a smaller share of the columns
    if kind == "solve":
        vec = 4 * (case["region"] or atoms)
        per = case["nu"] ** 2 * vec * (4.0 if case["precision"] == "fp64" else 1.0) + 60.0 * case["nu"] ** 3
        while 4 * atoms / case["share"] * per > 0.7 * 16384 * (30 ** 2 * 16384 + 60.0 * 30 ** 3):
            case["share"] *= 2
    return case


def _atoms(case):
    return {"diamond": 8 * case["size"] ** 3, "polymer": 69 * case["size"] + 2}.get(case["structure"], case["size"])


def _system(case, seed, size=None, structure_seed=0):
    size = case["size"] if size is None else size
    if case["structure"] == "diamond":
        t = tbsynth.build_tb(tbsynth.diamond(size, seed=structure_seed), check_spd=False)
    elif case["structure"] == "polymer":
        t = tbsynth.polymer_system(size, seed=structure_seed, check_spd=False)
    else:
        t = tbsynth.amorphous_system(size, seed=structure_seed, check_spd=False)
    # on-site energies N(0, 0.5 eV) per atom; every pair's hoppings and overlaps by about 2 percent
    rng = np.random.default_rng(seed)
    row, col = np.repeat(np.arange(t.n_block_rows), np.diff(t.row_ptr)), t.col_idx.astype(np.int64)
    pair, which = np.unique(np.minimum(row, col) * t.n_block_rows + np.maximum(row, col), return_inverse=True)
    f = 1.0 + 0.02 * rng.standard_normal(pair.size)[which]
    f[row == col] = 1.0
    t.H = t.H * f[:, None, None]
    t.S = t.S * f[:, None, None]
    real = t.orbital_mask.reshape(-1, 4).astype(float)
    shift = 0.5 * rng.standard_normal(t.n_block_rows)
    t.H[row == col] += (shift[:, None] * real)[:, :, None] * np.eye(4)
    return t


def _requests(case, seed):
    return [_system(case, seed + 1000 * q, n, structure_seed=q) for q, n in enumerate(_serve_sizes(case))]


def _serve_sizes(case):
    """Sizes of a serve case's requests: from half of `size` to twice it."""
    if case["structure"] == "polymer":
        return [case["size"] + q % 3 for q in range(case["requests"])]
    return [max(40, int(case["size"] * 2.0 ** (((5 * q) % 9) / 4.0 - 1.0))) for q in range(case["requests"])]


def _columns(case, t):
    """A rank's share of the real columns: those of a run of consecutive atoms (None: every column)."""
    if case["share"] == 1:
        return None
    atoms = np.arange(t.n_block_rows)
    n = max(1, t.n_block_rows // case["share"])
    a0 = (t.n_block_rows - n) // 2
    cols = t.real_columns()
    return cols[(cols >= 4 * atoms[a0]) & (cols < 4 * (a0 + n))]


def _shifts(case):
    """A half circle above the real axis around the occupied levels near the Fermi energy."""
    th = math.pi * (np.arange(case["shifts"]) + 0.5) / case["shifts"]
    return -6.0 + 10.0 * np.cos(th) + 1j * (0.3 + 10.0 * np.sin(th))


# the shared Fermi level that a rank's share is solved at (eV, near each kind's own)
MU_SHARE = {"diamond": 0.5, "amorphous": 4.0, "polymer": 1.8}


def prepare(case, seed):
    prec = PRECISION[case["precision"]]
    if case["kind"] == "serve":
        return {"case": case, "systems": _requests(case, seed), "server": m.Server(workers=4, hbm_budget_bytes=16 << 30)}
    t = _system(case, seed)
    state = {"case": case, "system": t}
    if case["kind"] == "request":
        return state
    state["ctx"] = m.setup_system(t, prec)
    state["columns"] = _columns(case, t)
    if case["kind"] == "outputs":
        m.marnoldi_solve(state["ctx"], None, case["nu"], case["region"], t.n_electrons, case["kT"])
        state["derivatives"] = tbsynth.build_tb_derivatives(t)
        state["shifts"] = _shifts(case)
    else:
        state["rho"] = torch.empty(t.nnzb, 4, 4, dtype=torch.float64, device="cuda")
        state["rhoE"] = torch.empty_like(state["rho"])
    return state


def run(state):
    case = state["case"]
    if case["kind"] == "serve":
        srv, prec = state["server"], PRECISION[case["precision"]]
        ids = [srv.submit_system(t, prec, case["nu"], case["region"], None, case["kT"]) for t in state["systems"]]
        got = [srv.wait(i) for i in ids]
        return {"rho": np.concatenate([g["rho"] for g in got]), "rhoE": np.concatenate([g["rhoE"] for g in got]),
                "energy": np.array([[g["band_energy"], g["mu"], g["N"]] for g in got])}
    t = state["system"]
    if case["kind"] == "request":
        ctx = m.setup_system(t, PRECISION[case["precision"]])
        m.marnoldi_solve(ctx, None, case["nu"], case["region"], t.n_electrons, case["kT"])
        rho, rhoE = m.marnoldi_density(ctx)
        energy = m.marnoldi_energy(ctx)
        m.marnoldi_destroy(ctx)
        return {"rho": rho, "rhoE": rhoE, "energy": np.array(energy)}
    ctx = state["ctx"]
    if case["kind"] == "outputs":
        dH, dS = state["derivatives"]
        return {"forces": m.marnoldi_forces(ctx, dH, dS), "green": m.marnoldi_green(ctx, state["shifts"])}
    if state["columns"] is None:
        m.marnoldi_solve(ctx, None, case["nu"], case["region"], t.n_electrons, case["kT"])
    else:
        m.marnoldi_solve(ctx, state["columns"], case["nu"], case["region"], 0.0, case["kT"],
                         mu_fixed=MU_SHARE[case["structure"]])
    m.marnoldi_density_device(ctx, state["rho"], state["rhoE"])
    return {"rho": state["rho"], "rhoE": state["rhoE"], "energy": np.array(m.marnoldi_energy(ctx))}


# ---------------------------------------------------------------- work
def work(case):
    """Flops of the Krylov build over the vectors' supports (the atoms within i hops of the column's atom, about
    5 i^3 of them in these solids and 16 i along a chain), the subspace eigenproblems and the output columns;
    bytes of H, S and of the results."""
    if case["kind"] == "serve":
        sizes = [_atoms({**case, "size": s}) for s in _serve_sizes(case)]
    else:
        sizes = [_atoms(case)]
    blocks = {"diamond": 15.4, "polymer": 7.0}.get(case["structure"], 11.25)
    real = 2.26 if case["structure"] == "polymer" else 4.0
    nbytes = flops = 0.0
    for n in sizes:
        cols = real * n / case["share"]
        nu, n_vec = case["nu"], min(n, case["region"] or n)
        out_bytes = 2 * 128.0 * blocks * cols / 4
        if case["kind"] == "outputs":
            nz = case["shifts"]
            nbytes += 2 * 3 * 128.0 * blocks * n + 24.0 * n + nz * 256.0 * blocks * n + 8.0 * cols * (4 * blocks + 2) * nu
            flops += cols * 4 * blocks * nu * (4.0 + 4.0 * nz)
            continue
        grow = (lambda i: 16.0 * i + 1) if case["structure"] == "polymer" else (lambda i: 5.0 * i ** 3 + 1)
        sup = [min(float(n_vec), grow(i + 1)) for i in range(nu)]
        krylov = sum(2 * 32.0 * blocks * s for s in sup)                        # H x and S x
        krylov += sum(8.0 * 4 * s * (nu - i) for i, s in enumerate(sup))        # three dots and a subtraction
        eig = 8.0 / 3.0 * nu ** 3 + 2.0 * (4 * blocks + 2) * nu ** 2
        flops += cols * (krylov + eig + 4.0 * 4 * blocks * nu)
        nbytes += 2 * 128.0 * blocks * n + out_bytes
    return {"bytes": nbytes, "flops": flops}


# ---------------------------------------------------------------- the same results in 64 bits, plain torch
def exact(case, seed):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    if case["kind"] == "serve":
        got = [_exact_one(case, t, dev) for t in _requests(case, seed)]
        return {"rho": np.concatenate([g["rho"] for g in got]), "rhoE": np.concatenate([g["rhoE"] for g in got]),
                "energy": np.stack([g["energy"] for g in got])}
    return _exact_one(case, _system(case, seed), dev)


def _fermi(x):
    e = torch.exp(-x.abs())
    return torch.where(x >= 0, e / (1 + e), 1 / (1 + e))


def _regions(t, n_reg):
    """The n_reg atoms nearest each atom by minimum-image distance (ties to the lower index), ascending."""
    pos, box = t.structure.positions, t.structure.box
    pos = np.mod(pos, box)
    out = np.empty((t.n_block_rows, n_reg), np.int64)
    for j in range(t.n_block_rows):
        d = pos - pos[j]
        d -= box * np.rint(d / box)
        d2 = (d[:, 0] ** 2 + d[:, 1] ** 2) + d[:, 2] ** 2
        near = np.flatnonzero(d2 <= np.partition(d2, n_reg - 1)[n_reg - 1])
        out[j] = np.sort(near[np.argsort(d2[near], kind="stable")[:n_reg]])
    return out


def _exact_one(case, t, dev):
    nu, kT, M = case["nu"], case["kT"], t.M
    f64 = dict(dtype=torch.float64, device=dev)
    H, S = torch.as_tensor(t.H, **f64), torch.as_tensor(t.S, **f64)
    rp, ci = t.row_ptr, t.col_idx.astype(np.int64)
    row = np.repeat(np.arange(t.n_block_rows), np.diff(rp))
    a4 = np.arange(4)
    ri = torch.as_tensor(np.broadcast_to(4 * row[:, None, None] + a4[:, None], (row.size, 4, 4)).reshape(-1), device=dev)
    cj = torch.as_tensor(np.broadcast_to(4 * ci[:, None, None] + a4, (row.size, 4, 4)).reshape(-1), device=dev)
    idx = torch.stack([ri, cj])
    Hs = torch.sparse_coo_tensor(idx, H.reshape(-1), (M, M)).to_sparse_csr()
    Ss = torch.sparse_coo_tensor(idx, S.reshape(-1), (M, M)).to_sparse_csr()
    Sdiag = S[torch.as_tensor(np.flatnonzero(row == ci), device=dev)].diagonal(dim1=1, dim2=2).reshape(-1)
    cols = _columns(case, t)
    cols = t.real_columns() if cols is None else cols
    reg = _regions(t, case["region"]) if case["region"] else None
    m_vec = 4 * (case["region"] or t.n_block_rows)
    chunk = int(max(1, min(cols.size, 24e9 / (8.0 * (2.2 * nu * m_vec + 6 * M)))))
    # the pattern rows of every column: atom I of block (I, J), whose mirror is stored at (J, I)
    maxrow = int(np.diff(rp).max())
    slot = np.arange(row.size) - rp[row]
    nbr = np.zeros((t.n_block_rows, maxrow), np.int64)
    blk = np.full((t.n_block_rows, maxrow), -1, np.int64)
    order = np.lexsort((row, ci))                       # blocks (I, J) by J, then I
    nbr[row, slot] = ci
    blk[ci[order], slot] = order                        # block (I, J) for the slot-th neighbour I of J
    eps, w, tt, P = [], [], [], []
    for c0 in range(0, cols.size, chunk):
        j = torch.as_tensor(cols[c0:c0 + chunk], device=dev)
        C = j.numel()
        at = torch.arange(C, device=dev)
        sel = None
        if reg is not None:
            r = torch.as_tensor(reg, device=dev)[j // 4]
            sel = (4 * r[:, :, None] + torch.arange(4, device=dev)).reshape(C, m_vec)

        def apply(A, x):
            if sel is None:
                return (A @ x.t()).t().contiguous()
            full = torch.zeros(C, M, **f64).scatter_(1, sel, x)
            return (A @ full.t()).t().gather(1, sel)

        jl = j if sel is None else (sel == j[:, None]).to(torch.int8).argmax(1)
        K = torch.zeros(C, nu, m_vec, **f64)
        SK = torch.zeros(C, nu, m_vec, **f64)
        K[at, 0, jl] = Sdiag[j].rsqrt()
        SK[:, 0] = apply(Ss, K[:, 0])
        A = torch.zeros(C, nu, nu, **f64)
        for n in range(nu):
            u = apply(Hs, K[:, n])
            A[:, :n + 1, n] = torch.bmm(K[:, :n + 1], u[:, :, None])[:, :, 0]
            if n + 1 == nu:
                break
            for _ in range(2):
                d = torch.bmm(SK[:, :n + 1], u[:, :, None])
                u = u - torch.bmm(K[:, :n + 1].transpose(1, 2), d)[:, :, 0]
            su = apply(Ss, u)
            s = (u * su).sum(1).rsqrt()[:, None]
            K[:, n + 1], SK[:, n + 1] = u * s, su * s
        del SK
        A = A.triu() + A.triu(1).transpose(1, 2)
        e, V = torch.linalg.eigh(A)
        q = K[at, :, jl]
        tq = (V * q[:, :, None]).sum(1)
        eps.append(e)
        tt.append(tq)
        w.append(Sdiag[j].sqrt()[:, None] * V[:, 0] * tq)
        atom = torch.as_tensor(nbr[cols[c0:c0 + chunk] // 4], device=dev)        # C, maxrow
        if sel is None:
            ra, inside = atom, torch.ones_like(atom, dtype=torch.bool)
        else:
            ra = torch.searchsorted(r, atom).clamp(max=case["region"] - 1)
            inside = r.gather(1, ra) == atom
        pos = (4 * ra[:, :, None] + torch.arange(4, device=dev)).reshape(C, 4 * maxrow)
        Kp = K.gather(2, pos[:, None, :].expand(C, nu, 4 * maxrow)) * inside.repeat_interleave(4, 1)[:, None, :]
        P.append(torch.bmm(Kp.transpose(1, 2), V))
        del K, Kp, V
    eps, w, tt, P = torch.cat(eps), torch.cat(w), torch.cat(tt), torch.cat(P)

    def scatter(y):
        """The columns P y on the block pattern."""
        v = torch.bmm(P.to(y.dtype), y[:, :, None])[:, :, 0].reshape(cols.size, maxrow, 4)
        out = torch.zeros(row.size, 4, 4, dtype=y.dtype, device=dev)
        b = torch.as_tensor(blk[cols // 4], device=dev)
        ok = b >= 0
        cb = torch.as_tensor(cols % 4, device=dev)[:, None].expand_as(b)
        out[b[ok], :, cb[ok]] = v[ok]
        return out

    def count(mu):
        return float((2 * _fermi((eps - mu) / kT) * w).sum())

    if case["share"] == 1:
        lo, hi, ne = float(eps.min()) - 40 * kT, float(eps.max()) + 40 * kT, t.n_electrons
        for _ in range(200):
            mu = 0.5 * (lo + hi)
            n = count(mu)
            if abs(n - ne) <= 1e-12 * ne:
                break
            lo, hi = (mu, hi) if n < ne else (lo, mu)
    else:
        mu = MU_SHARE[case["structure"]]
    f2 = 2 * _fermi((eps - mu) / kT)
    rho, rhoE = scatter(f2 * tt), scatter(f2 * eps * tt)
    if case["kind"] == "outputs":
        dH, dS = (torch.as_tensor(x, **f64) for x in tbsynth.build_tb_derivatives(t))
        tr = torch.as_tensor(blk[row, slot], device=dev)                         # block (J, I) of block (I, J)
        rb, reb = (rho + rho[tr].transpose(1, 2)) / 2, (rhoE + rhoE[tr].transpose(1, 2)) / 2
        per = 2 * (rb * dH - reb * dS).sum((2, 3)) * torch.as_tensor(row != ci, device=dev)
        F = torch.zeros(t.n_block_rows, 3, **f64).index_add_(0, torch.as_tensor(row, device=dev), per.t().contiguous())
        z = torch.as_tensor(_shifts(case), device=dev)
        G = torch.stack([scatter(tt / (x - eps)) for x in z])
        return {"forces": F.cpu().numpy(), "green": G.cpu().numpy()}
    energy = np.array([float((f2 * eps * w).sum()), mu, count(mu)])
    return {"rho": rho.cpu().numpy(), "rhoE": rhoE.cpu().numpy(), "energy": energy}
