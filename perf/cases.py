"""The calls whose speed matters: what a program that uses the library has it do, through its public
entry points, from one small block to a full mesh.

A case is a dict of plain values:
  kind    apply      ghost exchange + the requested centred derivatives of every field
          advect     ghost exchange + the upwinded shift-advection term of every field
          wave       one classical RK4 step of the wave system
          shiftwave  one 2S low-storage step of the shifted wave system with dissipation
          advstep    one 2S low-storage step of the advection equation with dissipation
  nbx, nby, nbz, N   periodic box of nbx x nby x nbz blocks of N^3 ("apply" also has mesh = "levels":
                     448 blocks of 16^3 and 64 of 32^3 at a 2:1 refined octant)
  nf, dtype, prec, n_iter, ops, scheme   fields, their type, the arithmetic (tc: tensor-core exact
                     slices, fp64: banded solves), hybrid iterations, "all" nine ops or some, Q13 or P12

Fields are sums of plane waves that the mesh resolves with at least 8 points per wavelength, with
Gaussian bumps beside them; the two-level mesh has the inverse-distance fields of a puncture data set.
``exact`` restates each call with dense block operators in 64-bit torch.
"""
import math

import numpy as np
import torch

from paper_2302_14858_gb300 import cfd
from paper_2302_14858_gb300 import workloads as W

G = 4  # ghost layers
OPS = ("dx", "dy", "dz", "dxx", "dyy", "dzz", "dxy", "dxz", "dyz")
PREC = {"tc": cfd.CFD_TC_BF16_EXACT, "fp64": cfd.CFD_FP64_BANDED}

# Interior and closure stencils: the tuned Q^1_3[1] (first and second degree) and the Pade P^1_2.
Q13_1 = dict(deriv=1, order=6, a=0.3798792289490848,
             rhs=[0.002327294780787575, -0.052602255439511914, -0.7816566024124237, 0.0, 0.7816566024124237,
                  0.052602255439511914, -0.002327294780787575],
             closure=[0.0035978349494889122, -0.038253676363600136, 0.20036968929284477, -0.8003696892928448, 0.0,
                      0.8003696892928448, -0.20036968929284477, 0.038253676363600136, -0.0035978349494889122])
Q13_2 = dict(deriv=2, order=6, a=0.24246602513914975,
             rhs=[-0.0037062570918369297, 0.1409592301669797, 0.954451443436913, -2.1834088330241115,
                  0.954451443436913, 0.1409592301669797, -0.0037062570918369297],
             closure=[-0.00181426951185116, 0.025625267205920392, -0.20079954633183247, 1.601599092663665,
                      -2.8492210880518036, 1.601599092663665, -0.20079954633183247, 0.025625267205920392,
                      -0.00181426951185116])
P12_1 = dict(deriv=1, order=6, a=1.0 / 3.0, rhs=[-1.0 / 36, -28.0 / 36, 0.0, 28.0 / 36, 1.0 / 36],
             closure=[1.0 / 300, -11.0 / 300, 59.0 / 300, -239.0 / 300, 0.0, 239.0 / 300, -59.0 / 300, 11.0 / 300,
                      -1.0 / 300])
P12_2 = dict(deriv=2, order=6, a=2.0 / 11.0, rhs=[3.0 / 44, 48.0 / 44, -102.0 / 44, 48.0 / 44, 3.0 / 44],
             closure=[-0.0014814814814814814, 0.022962962962962963, -0.19148148148148147, 1.582962962962963,
                      -2.825925925925926, 1.582962962962963, -0.19148148148148147, 0.022962962962962963,
                      -0.0014814814814814814])
SCHEMES = {"Q13": (Q13_1, Q13_2), "P12": (P12_1, P12_2)}
# The upwind scheme X_2 with its closure; it iterates on the node next to the block.
X2 = dict(order=6, a=407.0 / 600, lo=-4, c_sup=407.0 / 600, c_lo=-4, kc=1,
          rhs=[-0.0007678571428571428, 0.012087301587301588, -0.14283333333333334, -1.1026944444444444,
               0.8506944444444444, 0.4538333333333333, -0.08105555555555556, 0.011503968253968254,
               -0.0007678571428571428],
          closure=[0.0011438791712845284, -0.014257076205437428, 0.08954362614392307, -0.4677486551986694,
                   -0.8386567259077224, 1.0994919901690046, 0.13907812667610517, -0.007953566088123195,
                   -0.0008966670363147505, 0.0002550682759499099])
# Four-stage, fourth-order 2S low-storage Runge-Kutta (gamma1, gamma2, beta, delta).
RK2S = ([0.0, 0.068841064670197562, 0.62754761399692844, -0.59911219706265022],
        [1.0, 0.81058824734452378, 1.3891900984667538, 1.2610225117075399],
        [1.2299693289723146, 0.079894519849001553, 0.93225854169045408, 0.45482163406909008],
        [1.0, 0.14874467817694941, -0.88063710498437737, 1.0])
SIGMA, KO_R = 0.04, 4           # Kreiss-Oliger strength and order
SHIFT = (0.3, -0.2, 0.1)        # constant shift of the shifted wave
ADV_DIR = (math.cos(math.pi / 6), math.sin(math.pi / 6))  # advection direction: 30 degrees


def _case(kind, nb, N, **more):
    nbx, nby, nbz = (nb, nb, nb) if isinstance(nb, int) else nb
    c = dict(kind=kind, nbx=nbx, nby=nby, nbz=nbz, N=N, nf=1, dtype="f64", prec="tc", n_iter=0, ops="all",
             scheme="Q13", mesh="box")
    c.update(more)
    return c


def listed():
    return [
        # the smallest call: one periodic line mesh of one block, d_x of one field
        _case("apply", 1, 32, name="line32_dx_tc", ops="dx", scheme="P12"),
        # a small job in plain FP64 with one iteration (27 blocks, odd counts): test and set-up runs
        _case("apply", 3, 16, name="cube48_fp64_it1", prec="fp64", n_iter=1),
        # a small mesh on the tensor cores: 64 blocks of 16^3, two fields
        _case("apply", 4, 16, name="cube64_b16_f2_tc", nf=2),
        # the ordinary small-block mesh: 512 blocks of 16^3, four fields
        _case("apply", 8, 16, name="grid128_b16_f4_tc", nf=4),
        # the full mesh: 512 blocks of 32^3, four fields, closed blocks
        _case("apply", 8, 32, name="grid256_b32_f4_tc", nf=4),
        # the same with the one hybrid iteration that production runs use
        _case("apply", 8, 32, name="grid256_b32_f4_tc_it1", nf=4, n_iter=1),
        # the 22 single-precision fields of an evolution system on a two-level mesh
        _case("apply", 8, 16, name="levels_f22_f32_tc", mesh="levels", nf=22, dtype="f32"),
        # plain FP64 with one iteration on the small-block mesh: the accuracy runs
        _case("apply", 8, 16, name="grid128_b16_f4_fp64_it1", nf=4, prec="fp64", n_iter=1),
        # the upwinded shift terms of four fields on the full mesh
        _case("advect", 8, 32, name="advect256_b32_f4_tc_it1", nf=4, n_iter=1),
        # time steps of the wave and shifted-wave systems on the full mesh
        _case("wave", 8, 32, name="wave256_b32_rk4_tc"),
        _case("shiftwave", 8, 32, name="shiftwave256_b32_tc_it1", n_iter=1),
        # a step of the two-dimensional advection test: 144 small blocks, one block thick
        _case("advstep", (12, 12, 1), 16, name="adv2d192_b16_fp64_it1", prec="fp64", n_iter=1),
    ]


def draw(rng):
    kind = rng.choice(["apply"] * 6 + ["advect"] * 2 + ["wave", "shiftwave", "advstep"])
    prec = rng.choice(["tc", "tc", "fp64"])
    N = rng.choice([16, 32])
    top = 8 if N == 32 else 12
    nb = tuple(int(round(math.exp(rng.uniform(0.0, math.log(top))))) for _ in range(3))
    if kind == "advstep":
        nb = (nb[0], nb[1], 1)
    dtype = rng.choice(["f64", "f32"]) if kind in ("apply", "advect") else "f64"
    nf = int(round(math.exp(rng.uniform(0.0, math.log(22))))) if kind in ("apply", "advect") else 1
    n_iter = rng.choice([0, 1, 1, 2])
    ops = rng.choice(["all", "all", "first", "second", "dx"]) if kind == "apply" else "all"
    c = _case(kind, nb, N, nf=nf, dtype=dtype, prec=prec, n_iter=n_iter, ops=ops,
              scheme=rng.choice(["Q13", "Q13", "P12"]))
    # no more than the largest listed calls of its arithmetic
    most = (4 * 256 ** 3 if prec == "tc" else 6 * 128 ** 3) // (4 if kind == "shiftwave" else 1)
    while c["nf"] * _points(c) > most:
        if c["nf"] > 1:
            c["nf"] = (c["nf"] + 1) // 2
        else:
            k = max(("nbx", "nby", "nbz"), key=lambda a: c[a])
            c[k] = (c[k] + 1) // 2
    return c


def _points(c):
    if c["mesh"] == "levels":
        return 448 * 16 ** 3 + 64 * 32 ** 3
    return c["nbx"] * c["nby"] * c["nbz"] * c["N"] ** 3


def _ops(c):
    return {"all": OPS, "first": OPS[:3], "second": OPS[3:6], "dx": OPS[:1]}[c["ops"]]


def work(case):
    pts, nf, es = _points(case), case["nf"], 4 if case["dtype"] == "f32" else 8
    solve, biased = 19.0, 22.0  # operations of one banded solve, and of one upwinded derivative, per point
    if case["kind"] == "apply":
        ops = _ops(case)
        fl = sum(2 * solve if o in OPS[6:] else solve for o in ops)
        return {"bytes": pts * nf * es * (1 + len(ops)), "flops": pts * nf * fl}
    if case["kind"] == "advect":
        return {"bytes": pts * es * (2 * nf + 3), "flops": pts * nf * 3 * biased}
    if case["kind"] == "wave":
        return {"bytes": pts * 8 * 4, "flops": pts * 4 * (3 * solve + 10)}
    if case["kind"] == "shiftwave":
        return {"bytes": pts * 8 * 7, "flops": pts * 4 * (3 * solve + 6 * biased + 2 * 3 * 19 + 12)}
    return {"bytes": pts * 8 * (2 * nf + 3), "flops": pts * nf * 4 * (3 * biased + 3 * 19 + 6)}


# ---------------------------------------------------------------- inputs


def _mesh(c):
    if c["mesh"] == "levels":
        return W.box_in_box_mesh(G)
    return W.periodic_box_mesh(c["nbx"], c["nby"], c["nbz"], c["N"], G)


def _groups(mesh):
    """Runs of blocks of one size: (first block, number of blocks, N)."""
    out, b = [], 0
    n = [int(v) for v in mesh.n]
    while b < len(n):
        e = b
        while e < len(n) and n[e] == n[b]:
            e += 1
        out.append((b, e - b, n[b]))
        b = e
    return out


def _dev():
    return torch.device("cuda", torch.cuda.current_device())


def _coords(mesh, b0, nb, N):
    """Ghost-extended coordinates of blocks b0 .. b0+nb-1: (x, y, z), each [nb, E]."""
    loc = torch.arange(-G, N + G, dtype=torch.float64, device=_dev()) + 0.5
    o = torch.as_tensor(np.asarray(mesh.origin[b0:b0 + nb], np.float64), device=_dev())
    h = torch.as_tensor(np.asarray(mesh.dx[b0:b0 + nb], np.float64), device=_dev())
    return tuple((o[:, a:a + 1] + loc) * h[:, a:a + 1] for a in range(3))


def _box(mesh, c):
    """Period and points of the box along x, y, z."""
    if c["mesh"] == "levels":
        return (2 * math.pi,) * 3, (128,) * 3
    pts = (c["nbx"] * c["N"], c["nby"] * c["N"], c["nbz"] * c["N"])
    return tuple(float(p * mesh.dx[0, a]) for a, p in enumerate(pts)), pts


def _modes(r, box, pts, n=8):
    """Plane waves periodic in the box: integer wave numbers up to points / 8 per axis, either sign."""
    top = np.maximum(1, np.asarray(pts) // 8)
    k = np.stack([r.integers(-t, t + 1, size=n) for t in top], 1)
    k[(k == 0).all(1)] = 1
    return 2 * math.pi * k / np.asarray(box), r.uniform(-1, 1, n), r.uniform(0, 2 * math.pi, n)


def _waves(xyz, k, A, phase):
    """sum_j A_j sin(k_j . x + phase_j) on every point of every block: [nb, E, E, E]."""
    x, y, z = xyz
    kt = torch.as_tensor(k, device=x.device)
    At, pt = torch.as_tensor(A, device=x.device), torch.as_tensor(phase, device=x.device)
    zy = z[:, :, None, None] * kt[:, 2] + y[:, None, :, None] * kt[:, 1] + pt
    zy = torch.cat([At * torch.sin(zy), At * torch.cos(zy)], -1)          # [nb, z, y, 2n]
    kx = x[:, None, :] * kt[:, 0][None, :, None]
    nb, E = x.shape
    return torch.bmm(zy.reshape(nb, E * E, -1), torch.cat([torch.cos(kx), torch.sin(kx)], 1)).reshape(nb, E, E, E)


def _bump(xyz, centre, sigma, box):
    """A periodic Gaussian bump."""
    f = []
    for v, c0, L in zip(xyz, centre, box):
        f.append(sum(torch.exp(-(v - c0 - s * L) ** 2 / (2 * sigma ** 2)) for s in (-1, 0, 1)))
    return f[2][:, :, None, None] * f[1][:, None, :, None] * f[0][:, None, None, :]


def _punctures(xyz, centres):
    """sum_p 1 / (|x - x_p| + 1/2), distances to the nearest image in [0, 2 pi)^3."""
    out = 0.0
    for c0 in centres:
        d = []
        for v, cc in zip(xyz, c0):
            m = torch.remainder((v - cc).abs(), 2 * math.pi)
            d.append(torch.minimum(m, 2 * math.pi - m) ** 2)
        out = out + 1.0 / (torch.sqrt(d[2][:, :, None, None] + d[1][:, None, :, None] + d[0][:, None, None, :]) + 0.5)
    return out


def _dtype(c):
    return torch.float32 if c["dtype"] == "f32" else torch.float64


def _fields(mesh, c, r):
    """All fields on the ghost-extended blocks: flat, [block][field][E^3]."""
    box, pts = _box(mesh, c)
    what = []
    for q in range(c["nf"]):
        m = _modes(r, box, pts)
        what.append((m, r.uniform(0, 1, (2, 3))))
    out = []
    for b0, nb, N in _groups(mesh):
        xyz, E = _coords(mesh, b0, nb, N), N + 2 * G
        buf = torch.empty((nb, c["nf"], E, E, E), dtype=_dtype(c), device=_dev())
        for q, (m, u) in enumerate(what):
            if c["mesh"] == "levels":
                buf[:, q] = (_waves(xyz, *m) + _punctures(xyz, 2 * math.pi * u)).to(buf.dtype)
            elif q % 2 == 0:
                buf[:, q] = _waves(xyz, *m).to(buf.dtype)
            else:
                buf[:, q] = (0.25 * _waves(xyz, *m) + _bump(xyz, [a * L for a, L in zip(u[0], box)], 0.1 * max(box),
                                                            box)).to(buf.dtype)
        out.append(buf.reshape(-1))
    return torch.cat(out) if len(out) > 1 else out[0]


def _shift_fields(mesh, c):
    """(beta^x, beta^y, beta^z): both signs inside every block, or the constant vectors of the steps."""
    (b0, nb, N), = _groups(mesh)
    x, y, z = _coords(mesh, b0, nb, N)
    E = N + 2 * G
    buf = torch.empty((nb, 3, E, E, E), dtype=_dtype(c), device=_dev())
    if c["kind"] == "advect":
        X, Y, Z = x[:, None, None, :], y[:, None, :, None], z[:, :, None, None]
        buf[:, 0] = (torch.cos(X + 2 * Z) + 0.1).to(buf.dtype)
        buf[:, 1] = torch.sin(Y - X).to(buf.dtype)
        buf[:, 2] = (0.5 * torch.cos(3 * Y) * torch.sin(Z)).to(buf.dtype)
    else:
        v = SHIFT if c["kind"] == "shiftwave" else (-ADV_DIR[0], -ADV_DIR[1], 0.0)
        for a in range(3):
            buf[:, a] = v[a]
    return buf.reshape(-1)


def _wave_state(mesh, c, r):
    """Plane waves of the wave system: Phi and K = Phi_t at one time."""
    box, pts = _box(mesh, c)
    k, A, p = _modes(r, box, pts)
    w = np.sqrt((k ** 2).sum(1)) - (k @ np.asarray(SHIFT) if c["kind"] == "shiftwave" else 0.0)
    (b0, nb, N), = _groups(mesh)
    xyz = _coords(mesh, b0, nb, N)
    return _waves(xyz, k, A, p).reshape(-1), _waves(xyz, k, -A * np.sqrt((k ** 2).sum(1)) if c["kind"] != "shiftwave"
                                                    else -A * w, p + math.pi / 2).reshape(-1)


def _profile(mesh, c, r):
    """Smooth two-dimensional profiles of the advection step, constant along z: [block][field][E^3]."""
    box, pts = _box(mesh, c)
    (b0, nb, N), = _groups(mesh)
    x, y, z = _coords(mesh, b0, nb, N)
    E = N + 2 * G
    buf = torch.empty((nb, c["nf"], E, E, E), dtype=torch.float64, device=_dev())
    for q in range(c["nf"]):
        k, A, p = _modes(r, box, pts)
        k[:, 2] = 0.0
        u = r.uniform(0, 1, 2)
        buf[:, q] = 0.25 * _waves((x, y, z), k, A, p)
        g2 = _bump((x, y, torch.zeros_like(z)), (u[0] * box[0], u[1] * box[1], 0.0), 0.1 * max(box), (box[0], box[1], 1e9))
        buf[:, q] += g2
    return buf.reshape(-1)


def prepare(case, seed):
    c, r = case, np.random.Generator(np.random.PCG64(seed))
    mesh = _mesh(c)
    biased = c["kind"] in ("advect", "shiftwave", "advstep")
    d1, d2 = SCHEMES[c["scheme"]]
    scheme = cfd.cfd_scheme_create(d1, d2)
    if biased:
        cfd.cfd_scheme_set_biased(scheme, X2)
    blocks = cfd.cfd_blocks_bind(scheme, mesh.n, mesh.dx, mesh.neighbors, G,
                                 cfd.CFD_F32 if c["dtype"] == "f32" else cfd.CFD_F64)
    prec, it, nf, dx = PREC[c["prec"]], c["n_iter"], c["nf"], float(mesh.dx[0, 0])
    s = dict(c=c, scheme=scheme, blocks=blocks, prec=prec)
    pts = _points(c)
    if c["kind"] == "apply":
        ops = _ops(c)
        s.update(fields=_fields(mesh, c, r), mask=cfd.op_mask(ops),
                 out=torch.empty(pts * nf * len(ops), dtype=_dtype(c), device=_dev()))
        need = cfd.cfd_apply_workspace(blocks, nf, s["mask"], prec, it)
    elif c["kind"] == "advect":
        s.update(fields=_fields(mesh, c, r), beta=_shift_fields(mesh, c),
                 out=torch.empty(pts * nf, dtype=_dtype(c), device=_dev()))
        need = cfd.cfd_biased_workspace(blocks, nf, prec, it)
    elif c["kind"] == "advstep":
        s.update(u=_profile(mesh, c, r), beta=_shift_fields(mesh, c), dt=0.1 * dx)
        need = cfd.cfd_advect_lsrk_workspace(blocks, nf, prec, it)
    else:
        phi, K = _wave_state(mesh, c, r)
        s.update(phi=phi, K=K, dt=0.25 * dx)
        if c["kind"] == "shiftwave":
            s["beta"] = _shift_fields(mesh, c)
            need = cfd.cfd_shifted_wave_workspace(blocks, prec, it)
        else:
            need = cfd.cfd_wave_workspace(blocks, prec, it)
    s["work"] = torch.empty(max(need, 256), dtype=torch.uint8, device=_dev())
    return s


def _interior(buf, c):
    """The blocks' own points of a field buffer (a view)."""
    N, E = c["N"], c["N"] + 2 * G
    v = buf.view(c["nbx"] * c["nby"] * c["nbz"], c["nf"], E, E, E)
    return v[:, :, G:G + N, G:G + N, G:G + N]


def run(state):
    s, c = state, state["c"]
    B, prec, it, nf = s["blocks"], s["prec"], c["n_iter"], c["nf"]
    if c["kind"] == "apply":
        cfd.cfd_exchange_ghosts(B, s["fields"], nf)
        cfd.cfd_apply(B, s["fields"], nf, s["mask"], prec, it, s["out"], s["work"])
        return s["out"]
    if c["kind"] == "advect":
        cfd.cfd_exchange_ghosts(B, s["fields"], nf)
        cfd.cfd_advect(B, s["fields"], nf, s["beta"], prec, it, s["out"], s["work"])
        return s["out"]
    if c["kind"] == "wave":
        cfd.cfd_wave_rk_step(B, s["phi"], s["K"], s["dt"], prec, it, s["work"])
        return _interior(s["phi"], c), _interior(s["K"], c)
    if c["kind"] == "shiftwave":
        cfd.cfd_shifted_wave_lsrk_step(B, s["phi"], s["K"], s["beta"], s["dt"], RK2S, SIGMA, KO_R, prec, it, s["work"])
        return _interior(s["phi"], c), _interior(s["K"], c)
    cfd.cfd_advect_lsrk_step(B, s["u"], nf, s["beta"], s["dt"], RK2S, SIGMA, KO_R, prec, it, s["work"])
    return _interior(s["u"], c)


# ---------------------------------------------------------------- the same in 64-bit torch


def _centred(d, N, h, cyclic):
    """Dense block operators of a centred scheme: closed (or cyclic) [N, E], iterated [N, E] with the
    coefficients of the neighbours' values at rows N-2 (below) and 1 (above)."""
    E, a, M = N + 2 * G, d["a"], len(d["rhs"]) // 2
    sc = h ** -d["deriv"]

    def rows(ks, closed):
        A, Bm = np.zeros((len(ks), len(ks))), np.zeros((len(ks), E))
        for r, k in enumerate(ks):
            A[r, r] = 1
            end = closed and k in (0, N - 1)
            co = d["closure"] if end else d["rhs"]
            w = len(co) // 2
            if cyclic:
                A[r, (r - 1) % N] += a
                A[r, (r + 1) % N] += a
                for m in range(-w, w + 1):
                    Bm[r, G + (k + m) % N] += co[m + w]
                continue
            if not end:
                if r > 0:
                    A[r, r - 1] = a
                if r < len(ks) - 1:
                    A[r, r + 1] = a
            Bm[r, G + k - w:G + k + w + 1] = co
        return A, Bm

    A, Bm = rows(range(N), not cyclic)
    D0 = np.linalg.solve(A, Bm) * sc
    if cyclic:
        return D0, None, None, None
    A, Bm = rows(range(-1, N + 1), False)
    I = np.zeros((N + 2, 2))
    I[0, 0] = I[-1, 1] = -a
    X = np.linalg.solve(A, np.concatenate([Bm * sc, I], 1))[1:N + 1]
    return D0, X[:, :E], X[:, E], X[:, E + 1]


def _upwind(N, h, side, cyclic):
    """Dense operators of the left-biased scheme (side +1) or its mirror (-1): closed (or cyclic), iterated
    and the coefficients of the neighbour's value."""
    d, E, kc = X2, N + 2 * G, X2["kc"]

    def left(n_extra, closed):
        n = N + n_extra
        A, Bm = np.eye(n), np.zeros((n, E + 1))
        for r in range(n):
            k = r - n_extra
            if n_extra and r == 0:
                Bm[r, E] = 1
                continue
            end = closed and k == 0
            co, lo = (d["closure"], d["c_lo"]) if end else (d["rhs"], d["lo"])
            if end:
                A[r, r + 1] += d["c_sup"]
            else:
                A[r, (r - 1) % n if cyclic else r - 1] += d["a"]
            for i, v in enumerate(co):
                j = k + lo + i
                Bm[r, G + (j % N if cyclic else j)] += v / h
        X = np.linalg.solve(A, Bm)[n_extra:]
        return X[:, :E], X[:, E]

    D0, _ = left(0, not cyclic)
    D1, cf = (None, None) if cyclic else left(kc, False)
    if side < 0:  # mirrored: points and rows reversed, the sign of the derivative too
        D0 = -D0[::-1, ::-1]
        D1, cf = (None, None) if D1 is None else (-D1[::-1, ::-1], cf[::-1])
    return D0, D1, cf


def _t(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device=_dev())


def _along(D, f, ax):
    """D applied along dimension ax of f (negative)."""
    if ax == -1:
        return torch.matmul(f, D.T)
    s = f.shape
    flat = f.reshape(*s[:ax], s[ax], -1)
    return torch.matmul(D, flat).reshape(*s[:ax], D.shape[0], *s[ax + 1:])


class _Blocks64:
    """The blocks of a box (or one level of a two-level mesh) and their operators, in float64."""

    def __init__(self, mesh, c, b0, nb, N):
        self.N, self.E, self.it = N, N + 2 * G, c["n_iter"]
        self.nbr = torch.as_tensor(np.where(mesh.neighbors[b0:b0 + nb] >= 0, mesh.neighbors[b0:b0 + nb] - b0, -1)
                                   .astype(np.int64), device=_dev())
        self.face = {a: tuple(self.nbr[:, W.DIRS.index(tuple(s if i == 3 + a else 0 for i in range(3)))]
                              for s in (-1, 1)) for a in (-1, -2, -3)}
        own = torch.arange(nb, device=_dev())
        self.cyc = {a: bool(((lo == own) & (hi == own)).all()) for a, (lo, hi) in self.face.items()}
        h, self.D, self.U, self.h = float(mesh.dx[b0, 0]), {}, {}, float(mesh.dx[b0, 0])
        for a in (-1, -2, -3):
            for d in SCHEMES[c["scheme"]]:
                self.D[a, d["deriv"]] = [None if v is None else _t(v) for v in _centred(d, N, h, self.cyc[a])]
            for s in (1, -1):
                self.U[a, s] = [None if v is None else _t(v) for v in _upwind(N, h, s, self.cyc[a])]

    def exchange(self, f):
        N = self.N
        for r, d in enumerate(W.DIRS):
            sel = (self.nbr[:, r] >= 0).nonzero()[:, 0]
            dst = tuple(slice(0, G) if v < 0 else slice(N + G, N + 2 * G) if v > 0 else slice(G, N + G) for v in d)
            src = tuple(slice(N, N + G) if v < 0 else slice(G, 2 * G) if v > 0 else slice(G, N + G) for v in d)
            if len(sel):
                f[(sel, slice(None)) + dst] = f[(self.nbr[sel, r], slice(None)) + src]
        return f

    def inner(self, f, keep=()):
        """The blocks' own points along every axis but those in keep."""
        return f[(Ellipsis,) + tuple(slice(None) if a in keep else slice(G, G + self.N) for a in (-3, -2, -1))]

    def deriv(self, f, ax, deg):
        """The decomposed derivative along ax of f, which has its ghosts along that axis."""
        D0, D1, cm, cp = self.D[ax, deg]
        out = _along(D0, f, ax)
        for _ in range(0 if D1 is None else self.it):
            lo, hi = self.face[ax]
            below, above = out.select(ax, self.N - 2)[lo].unsqueeze(ax), out.select(ax, 1)[hi].unsqueeze(ax)
            shape = [1] * out.dim()
            shape[ax] = self.N
            out = _along(D1, f, ax) + cm.reshape(shape) * below + cp.reshape(shape) * above
        return out

    def upwind(self, f, ax, side):
        D0, D1, cf = self.U[ax, side]
        out = _along(D0, f, ax)
        for _ in range(0 if D1 is None else self.it):
            lo, hi = self.face[ax]
            kc = X2["kc"]
            v = out.select(ax, self.N - kc)[lo] if side > 0 else out.select(ax, kc - 1)[hi]
            shape = [1] * out.dim()
            shape[ax] = self.N
            out = _along(D1, f, ax) + cf.reshape(shape) * v.unsqueeze(ax)
        return out

    def op(self, f, name):
        ax = [{"x": -1, "y": -2, "z": -3}[v] for v in name[1:]]
        if len(ax) == 2 and ax[0] != ax[1]:
            return self.deriv(self.deriv(self.inner(f, ax), ax[1], 1), ax[0], 1)
        return self.deriv(self.inner(f, ax[:1]), ax[0], len(ax))

    def advection(self, f, beta):
        """sum_i beta^i d_i f, the right-biased derivative where beta^i > 0, the left-biased one where < 0."""
        out = 0.0
        for i, a in enumerate((-1, -2, -3)):
            b, g = self.inner(beta[:, i:i + 1]), self.inner(f, (a,))
            out = out + b.clamp(min=0) * self.upwind(g, a, -1) + b.clamp(max=0) * self.upwind(g, a, 1)
        return out

    def dissipation(self, f):
        r, out = KO_R, 0.0
        for a in (-1, -2, -3):
            g = self.inner(f, (a,))
            for m in range(2 * r + 1):
                w = -((-1) ** r) / 4.0 ** r * SIGMA / self.h * (-1) ** m * math.comb(2 * r, m)
                out = out + w * g.narrow(a, G + m - r, self.N)
        return out


def _put(f, B, v):
    B.inner(f).copy_(v)
    return f


def exact(case, seed):
    c = case
    s = prepare(c, seed)
    mesh = _mesh(c)
    if c["kind"] in ("apply", "advect"):
        outs, at = [], 0
        for b0, nb, N in _groups(mesh):
            B, E = _Blocks64(mesh, c, b0, nb, N), N + 2 * G
            n = nb * c["nf"] * E ** 3
            f = B.exchange(s["fields"][at:at + n].view(nb, c["nf"], E, E, E).double())
            at += n
            if c["kind"] == "advect":
                outs.append(B.advection(f, s["beta"].view(nb, 3, E, E, E).double()).reshape(-1))
                continue
            ops = _ops(c)
            out = torch.empty((nb, c["nf"], len(ops), N, N, N), dtype=torch.float64, device=_dev())
            for i, o in enumerate(ops):
                out[:, :, i] = B.op(f, o)
            outs.append(out.reshape(-1))
        return torch.cat(outs) if len(outs) > 1 else outs[0]
    (b0, nb, N), = _groups(mesh)
    B, E, dt = _Blocks64(mesh, c, b0, nb, N), N + 2 * G, s["dt"]
    shape = (nb, c["nf"], E, E, E)
    beta = s["beta"].view(nb, 3, E, E, E) if "beta" in s else None

    def laplacian(f):
        return sum(B.op(f, o) for o in OPS[3:6])

    if c["kind"] == "wave":
        f = s["phi"].view(shape).clone()
        p0, k0 = B.inner(f).clone(), B.inner(s["K"].view(shape)).clone()
        sp, sk, kp, acc_p, acc_k = p0, k0, k0, 0.0, 0.0
        for weight, step in ((1, 0.5), (2, 0.5), (2, 1.0), (1, None)):
            dp, dk = sk, laplacian(B.exchange(_put(f, B, sp)))
            acc_p, acc_k = acc_p + weight * dp, acc_k + weight * dk
            if step:
                sp, sk = p0 + step * dt * dp, k0 + step * dt * dk
        return p0 + dt / 6 * acc_p, k0 + dt / 6 * acc_k
    if c["kind"] == "shiftwave":
        fs = [s["phi"].view(shape).clone(), s["K"].view(shape).clone()]
    else:
        fs = [s["u"].view(shape).clone()]
    s2 = [torch.zeros_like(B.inner(f)) for f in fs]
    for g1, g2, be, de in zip(*RK2S):
        for f in fs:
            B.exchange(f)
        F = [B.dissipation(f) + B.advection(f, beta) for f in fs]
        if c["kind"] == "shiftwave":
            F[0] = F[0] + B.inner(fs[1])
            F[1] = F[1] + laplacian(fs[0])
        for f, acc, rate in zip(fs, s2, F):
            acc.add_(B.inner(f), alpha=de)
            _put(f, B, g1 * B.inner(f) + g2 * acc + be * dt * rate)
    got = [B.inner(f) for f in fs]
    return tuple(got) if c["kind"] == "shiftwave" else got[0]
