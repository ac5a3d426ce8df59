"""The exact tensor-core kernel's dispatch: every form it accepts against the FP64 banded solve.

The kernel has compiled-in addressing for four ghost layers and a general form for other widths, TMA
staging where a tile is an aligned box of the input and element copies elsewhere, row boxes for the
x outputs where they are aligned, and one or two operators (16, 32 or 64 rows) per launch.  Tolerances:
1e-7 of the largest output for FP64 fields (the contract of the exact slices; 2^-37 of sum |D f| times
the cancellation of the operator) and 2e-6 for FP32 fields (their rounding).
"""
import numpy as np
import pytest

from paper_2302_14858_gb300 import workloads as W
from tests.helpers import desc, rel_max

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    from paper_2302_14858_gb300 import build
    build.build()
    from paper_2302_14858_gb300 import cfd
    return cfd


def run(lib, B, fields, nf, mask, prec, n_iter, out_offset):
    import torch
    nops, nint = bin(mask).count("1"), sum(int(n) ** 3 for n in B.block_n)
    buf = torch.full((nint * nf * nops + 8,), float("nan"), dtype=fields.dtype, device=fields.device)
    out = buf[out_offset:out_offset + nint * nf * nops]
    work = torch.empty(max(lib.cfd_apply_workspace(B, nf, mask, prec, n_iter), 256), dtype=torch.uint8,
                       device=fields.device)
    lib.cfd_apply(B, fields, nf, mask, prec, n_iter, out, work)
    lib.cfd_sync_status(B)
    return out.cpu().numpy().reshape(len(B.block_n), nf, nops, -1)


@pytest.mark.parametrize("nb,N,g,dtype,nf,ops,n_iter,offset", [
    ((2, 1, 3), 16, 4, "f64", 1, ("dx",), 0, 0),                     # 16 operator rows; a cyclic axis
    ((2, 1, 3), 16, 4, "f64", 3, ("dx", "dxx", "dyz"), 1, 0),
    ((3, 2, 2), 16, 4, "f32", 2, ("dx", "dy", "dz", "dxx", "dyy", "dzz", "dxy", "dxz", "dyz"), 2, 0),
    ((2, 2, 2), 32, 4, "f64", 1, ("dx", "dxy"), 1, 1),               # unaligned buffers: element copies
    ((2, 2, 1), 32, 4, "f32", 3, ("dxx", "dz", "dxz", "dyz"), 0, 1),
    ((2, 2, 2), 32, 4, "f32", 1, ("dy", "dyy"), 1, 2),
    ((2, 2, 2), 16, 5, "f64", 2, ("dx", "dyy", "dzz", "dxy", "dxz", "dyz"), 0, 0),   # other ghost widths
    ((2, 3, 2), 16, 5, "f32", 1, ("dx", "dy", "dz", "dxy"), 1, 0),
    ((2, 2, 2), 16, 8, "f64", 1, ("dx", "dz", "dyy", "dyz"), 0, 0),  # no padding column left
    ((2, 2, 2), 32, 6, "f64", 1, ("dx", "dy", "dz", "dxx", "dxz"), 1, 0),
    ((2, 2, 2), 32, 8, "f32", 1, ("dx", "dyy", "dz"), 0, 1),
])
def test_every_form_matches_the_banded_solve(lib, nb, N, g, dtype, nf, ops, n_iter, offset):
    import torch
    mesh = W.periodic_box_mesh(*nb, N, g)
    # wave numbers in units of the box: every axis is periodic
    L = [nb[a] * N * mesh.dx[0, a] for a in range(3)]
    r = W.rng(77 + N + g + n_iter)
    fs = []
    for _ in range(nf):
        s = W.sine_sum(r, 6, 1, 4)
        s.k = 2 * np.pi * s.k / np.asarray(L)
        fs.append(s)
    flat = W.pack(W.sample(mesh, fs, np.float32 if dtype == "f32" else np.float64))
    dev = torch.device("cuda", 0)
    hold = torch.zeros(flat.size + 8, dtype=torch.float32 if dtype == "f32" else torch.float64, device=dev)
    fields = hold[offset:offset + flat.size]
    fields.copy_(torch.from_numpy(flat))
    s = lib.cfd_scheme_create(desc("Q13_1_d1"), desc("Q13_1_d2"))
    B = lib.cfd_blocks_bind(s, mesh.n, mesh.dx, mesh.neighbors, g, lib.CFD_F32 if dtype == "f32" else lib.CFD_F64)
    mask = lib.op_mask(ops)
    got = run(lib, B, fields, nf, mask, lib.CFD_TC_BF16_EXACT, n_iter, offset)
    want = run(lib, B, fields, nf, mask, lib.CFD_FP64_BANDED, n_iter, 0)
    tol = 2e-6 if dtype == "f32" else 1e-7
    for i, op in enumerate(lib.ops_in_mask(mask)):
        for q in range(nf):
            e = rel_max(got[:, q, i], want[:, q, i])
            assert e < tol, (op, q, e)


@pytest.mark.parametrize("nblk", [1, 3])
def test_rows_with_a_flat_operator_keep_their_accuracy(lib, nblk):
    """A scheme whose interior stencil is nearly flat (its rows sum to several times their largest
    entry): the row scale makes room for the level-0 sums.  Random fields, closed blocks, d_x."""
    import torch
    N, g = 32, 6
    mesh = W.periodic_box_mesh(nblk, 1, 1, N, g)
    M = 5
    rhs = [0.0] * (2 * M + 1)
    for m in range(1, M + 1):          # antisymmetric, consistent: sum m a_m = (1 + 2a) / 2
        rhs[M + m] = 1.0
    c = (1 + 2 * 0.45) / (2.0 * sum(m * rhs[M + m] for m in range(1, M + 1)))
    for m in range(1, M + 1):
        rhs[M + m] *= c
        rhs[M - m] = -rhs[M + m]
    d1 = {"deriv": 1, "order": 2, "a": 0.45, "rhs": rhs, "closure": rhs}
    s = lib.cfd_scheme_create(d1, None)
    B = lib.cfd_blocks_bind(s, mesh.n, mesh.dx, mesh.neighbors, g, lib.CFD_F64)
    E = N + 2 * g
    f = W.rng(5).uniform(-1, 1, size=(nblk, 1, E, E, E))
    dev = torch.device("cuda", 0)
    fields = torch.from_numpy(f.reshape(-1).copy()).to(dev)
    got = run(lib, B, fields, 1, lib.CFD_OP_DX, lib.CFD_TC_BF16_EXACT, 0, 0).reshape(nblk, N, N, N)
    # the closed (cyclic where the block is its own neighbour) system, solved in FP64
    A, Bm = np.eye(N), np.zeros((N, E))
    for k in range(N):
        if nblk == 1:
            A[k, (k - 1) % N] += 0.45
            A[k, (k + 1) % N] += 0.45
            for m in range(-M, M + 1):
                Bm[k, g + (k + m) % N] += rhs[m + M]
        else:
            if 0 < k < N - 1:
                A[k, k - 1] = A[k, k + 1] = 0.45
            Bm[k, g + k - M:g + k + M + 1] = rhs
    D = np.linalg.solve(A, Bm) / mesh.dx[0, 0]
    I = slice(g, g + N)
    want = np.einsum("ij,bzyj->bzyi", D, f[:, 0, I, I, :])
    bound = 2.0 ** -36 * np.abs(D).sum(1)      # |f| < 1 = tau; 2^-37 sum |D f| is the design bound
    assert np.all(np.abs(got - want) <= bound[None, None, None, :])


@pytest.mark.parametrize("N,g,dtype,nf,n_iter,offset", [
    (32, 4, "f64", 4, 0, 0),      # a quarter of a million points, four fields: the side is chosen in the stages
    (32, 4, "f64", 4, 1, 1),      # element copies in, per-thread x outputs
    (32, 4, "f32", 6, 2, 0),      # two groups of four fields, the second partial
    (16, 6, "f64", 5, 1, 0),      # another ghost width: run-time addressing
    (16, 4, "f32", 4, 0, 1),
])
def test_upwinded_stages_match_the_banded_solve(lib, N, g, dtype, nf, n_iter, offset):
    """The shift term where the stages store only the side that the shift selects, with shift components
    of both signs, of one sign and of zeros (of either sign, which select the same finite side)."""
    import torch
    from tests.helpers import SCHEMES
    nb = 64 // N
    mesh = W.periodic_box_mesh(nb, nb, nb, N, g)
    np_t, t_t = (np.float32, torch.float32) if dtype == "f32" else (np.float64, torch.float64)
    r = W.rng(300 + N + g + n_iter)
    fs = []
    for _ in range(nf + 1):
        s = W.sine_sum(r, 6, 1, 4)
        s.k = 2 * np.pi * s.k / (64 * mesh.dx[0, 0])
        fs.append(s)
    E = N + 2 * g
    flat = W.pack(W.sample(mesh, fs, np_t)).reshape(nb ** 3, nf + 1, E ** 3)
    fields = np.ascontiguousarray(flat[:, :nf]).reshape(-1)
    shift = np.zeros((nb ** 3, 3, E ** 3), np_t)
    shift[:, 0] = flat[:, nf]                                   # both signs inside a block
    shift[:, 1] = 0.25                                          # one side everywhere
    shift[:, 2] = np.where(np.arange(E ** 3) % 3 == 0, np_t(-0.0), np_t(0.0))
    shift[nb ** 3 // 2:, 2] = -0.5
    dev = torch.device("cuda", 0)

    def put(a):
        hold = torch.zeros(a.size + 8, dtype=t_t, device=dev)
        v = hold[offset:offset + a.size]
        v.copy_(torch.from_numpy(a.reshape(-1)))
        return v

    f, b = put(fields), put(shift)
    s = lib.cfd_scheme_create(desc("Q13_1_d1"), None)
    lib.cfd_scheme_set_biased(s, SCHEMES["X2_d1"])
    B = lib.cfd_blocks_bind(s, mesh.n, mesh.dx, mesh.neighbors, g, lib.CFD_F32 if dtype == "f32" else lib.CFD_F64)
    outs = []
    for prec in (lib.CFD_TC_BF16_EXACT, lib.CFD_FP64_BANDED):
        buf = torch.full((64 ** 3 * nf + 8,), float("nan"), dtype=t_t, device=dev)
        out = buf[offset:offset + 64 ** 3 * nf]
        work = torch.empty(max(lib.cfd_biased_workspace(B, nf, prec, n_iter), 256), dtype=torch.uint8, device=dev)
        lib.cfd_advect(B, f, nf, b, prec, n_iter, out, work)
        lib.cfd_sync_status(B)
        outs.append(out.double().cpu().numpy().reshape(nb ** 3, nf, -1))
    tol = 2e-6 if dtype == "f32" else 1e-7
    for q in range(nf):
        assert rel_max(outs[0][:, q], outs[1][:, q]) < tol, q


@pytest.mark.parametrize("N,g,offset", [(16, 4, 0), (16, 4, 1), (32, 4, 0), (32, 4, 1), (32, 5, 0)])
def test_wave_step_with_dissipation_matches_the_banded_one(lib, N, g, offset):
    """One 2S step with r = 4 dissipation (the FP32 ring of planes) on aligned and unaligned fields, for an
    odd ghost width and with an axis of a single block."""
    import torch
    from oracle import timestep as T
    mesh = W.periodic_box_mesh(2, 1, 2, N, g)
    L = [m * N * mesh.dx[0, a] for a, m in enumerate((2, 1, 2))]
    r = W.rng(900 + N + g)
    fs = []
    for _ in range(2):
        s = W.sine_sum(r, 6, 1, 4)
        s.k = 2 * np.pi * s.k / np.asarray(L)
        fs.append(s)
    E = N + 2 * g
    flat = W.pack(W.sample(mesh, fs, np.float64)).reshape(4, 2, E ** 3)
    dev = torch.device("cuda", 0)
    s = lib.cfd_scheme_create(desc("Q13_1_d1"), desc("Q13_1_d2"))
    B = lib.cfd_blocks_bind(s, mesh.n, mesh.dx, mesh.neighbors, g, lib.CFD_F64)
    outs = []
    for prec in (lib.CFD_TC_BF16_EXACT, lib.CFD_FP64_BANDED):
        u = []
        for q in range(2):
            hold = torch.zeros(4 * E ** 3 + 2, dtype=torch.float64, device=dev)
            v = hold[offset:offset + 4 * E ** 3]
            v.copy_(torch.from_numpy(flat[:, q].reshape(-1).copy()))
            u.append(v)
        work = torch.empty(lib.cfd_wave_lsrk_workspace(B, prec, 1), dtype=torch.uint8, device=dev)
        lib.cfd_wave_lsrk_step(B, u[0], u[1], 0.2 * mesh.dx.min(), T.lsrk2s_rk4_float(), 0.04, 4, prec, 1, work)
        lib.cfd_sync_status(B)
        I = slice(g, g + N)
        outs.append([v.cpu().numpy().reshape(4, E, E, E)[:, I, I, I] for v in u])
    for q in range(2):
        assert rel_max(outs[0][q], outs[1][q]) < 1e-7, q


@pytest.mark.parametrize("nb,N,nf,graph", [((1, 1, 1), 32, 1, False), ((2, 2, 2), 16, 1, False), ((2, 2, 2), 16, 1, True),
                                           ((4, 4, 4), 16, 3, False), ((5, 5, 5), 16, 2, False), ((4, 4, 4), 32, 2, False)])
def test_chained_launches_keep_their_order(lib, nb, N, nf, graph):
    """Exchanges and applies follow one another without a host synchronisation, each pass on fields that a
    torch kernel or the apply before it has just written or read: the same bits as with a synchronisation
    after every call.  Sizes on both sides of the line up to which an exchange is chained."""
    import torch
    g, dev = 4, torch.device("cuda", 0)
    mesh = W.periodic_box_mesh(*nb, N, g)
    E, nblk, mask = N + 2 * g, nb[0] * nb[1] * nb[2], lib.op_mask(("dx", "dyy", "dz", "dxz", "dyz", "dy"))
    s = lib.cfd_scheme_create(desc("Q13_1_d1"), desc("Q13_1_d2"))
    B = lib.cfd_blocks_bind(s, mesh.n, mesh.dx, mesh.neighbors, g, lib.CFD_F64)
    start = torch.from_numpy(W.rng(nblk + N).uniform(-1, 1, size=nblk * nf * E ** 3)).to(dev)
    passes, prec = 6, lib.CFD_TC_BF16_EXACT
    work = torch.empty(max(lib.cfd_apply_workspace(B, nf, mask, prec, 1), 256), dtype=torch.uint8, device=dev)

    def run(sync, fields, outs):
        for p in range(passes):
            lib.cfd_exchange_ghosts(B, fields, nf)
            if sync:
                torch.cuda.synchronize()
            lib.cfd_apply(B, fields, nf, mask, prec, 1, outs[p], work)
            if sync:
                torch.cuda.synchronize()
            if p % 2:            # every other pass follows the apply directly
                fields.mul_(-0.5)

    want = torch.zeros(passes, nblk * nf * 6 * N ** 3, dtype=torch.float64, device=dev)
    f = start.clone()
    run(True, f, want)
    got = torch.zeros_like(want)
    h = start.clone()
    torch.cuda.synchronize()
    if graph:
        G = torch.cuda.CUDAGraph()
        with torch.cuda.graph(G):
            run(False, h, got)
        h.copy_(start)
        got.zero_()
        G.replay()
    else:
        run(False, h, got)
    lib.cfd_sync_status(B)
    torch.cuda.synchronize()
    assert torch.equal(got, want) and torch.equal(h, f)


def interleaved(g, nf, seed, np_t):
    """Eight 16^3 and three 32^3 blocks, each size a periodic box of its own, in an order that keeps neither
    size's blocks together: (n, dx, neighbours, per-block samples of nf + 3 fields)."""
    from types import SimpleNamespace
    parts = []
    for k, (nb, N) in enumerate((((2, 2, 2), 16), ((1, 3, 1), 32))):
        mesh = W.periodic_box_mesh(*nb, N, g)
        L = [nb[a] * N * mesh.dx[0, a] for a in range(3)]
        r = W.rng(seed + k)
        fs = []
        for _ in range(nf + 3):
            s = W.sine_sum(r, 6, 1, 3)
            s.k = 2 * np.pi * s.k / np.asarray(L)
            fs.append(s)
        parts.append((mesh, W.sample(mesh, fs, np_t)))
    (a, fa), (b, fb) = parts
    order = np.array([0, 8, 1, 2, 3, 9, 4, 5, 10, 6, 7])    # position -> block of (a, b)
    where = np.argsort(order)
    nbr = np.concatenate([np.asarray(a.neighbors), np.asarray(b.neighbors) + 8])
    return SimpleNamespace(n=np.concatenate([a.n, b.n])[order], dx=np.concatenate([a.dx, b.dx])[order],
                           neighbors=where[nbr][order].astype(np.int32), fields=[(fa + fb)[i] for i in order])


@pytest.mark.parametrize("g,dtype,nf,n_iter,offset", [
    (4, "f64", 2, 0, 0), (4, "f64", 1, 1, 0), (4, "f32", 3, 0, 0), (4, "f32", 2, 1, 0), (4, "f64", 2, 0, 1),
    (5, "f64", 1, 0, 0), (6, "f32", 1, 0, 0),
])
def test_sizes_that_alternate_in_block_order(lib, g, dtype, nf, n_iter, offset):
    """Block ids of one size that are not consecutive: inputs staged by element or 16-byte copies, offsets from
    the tables, x outputs as row boxes of the whole output.  Apply against the banded solve, and (where the
    biased windows take the ghost width) the upwinded shift term."""
    import torch
    from tests.helpers import SCHEMES
    np_t, t_t = (np.float32, torch.float32) if dtype == "f32" else (np.float64, torch.float64)
    m = interleaved(g, nf, 500 + g + n_iter, np_t)
    dev = torch.device("cuda", 0)

    def put(a):
        hold = torch.zeros(a.size + 8, dtype=t_t, device=dev)
        v = hold[offset:offset + a.size]
        v.copy_(torch.from_numpy(np.ascontiguousarray(a, np_t)))
        return v

    fields = put(np.concatenate([b[:nf].reshape(-1) for b in m.fields]))
    shift = put(np.concatenate([b[nf:].reshape(-1) for b in m.fields]))
    s = lib.cfd_scheme_create(desc("Q13_1_d1"), desc("Q13_1_d2"))
    lib.cfd_scheme_set_biased(s, SCHEMES["X2_d1"])
    B = lib.cfd_blocks_bind(s, m.n, m.dx, m.neighbors, g, lib.CFD_F32 if dtype == "f32" else lib.CFD_F64)
    tol = 2e-6 if dtype == "f32" else 1e-7
    nint = sum(int(v) ** 3 for v in m.n)

    def call(what, prec, nops):
        buf = torch.full((nint * nf * nops + 8,), float("nan"), dtype=t_t, device=dev)
        out = buf[offset:offset + nint * nf * nops]
        if what == "apply":
            need = lib.cfd_apply_workspace(B, nf, lib.CFD_OP_ALL, prec, n_iter)
        else:
            need = lib.cfd_biased_workspace(B, nf, prec, n_iter)
        work = torch.empty(max(need, 256), dtype=torch.uint8, device=dev)
        if what == "apply":
            lib.cfd_apply(B, fields, nf, lib.CFD_OP_ALL, prec, n_iter, out, work)
        elif what == "advect":
            lib.cfd_advect(B, fields, nf, shift, prec, n_iter, out, work)
        else:
            lib.cfd_apply_biased(B, fields, nf, 7, 1, prec, n_iter, out, work)
        lib.cfd_sync_status(B)
        flat, at, per = out.double().cpu().numpy(), 0, {}
        for v in m.n:  # [size][op]: the group's blocks and fields
            k = nf * nops * int(v) ** 3
            per.setdefault(int(v), []).append(flat[at:at + k].reshape(nf, nops, -1))
            at += k
        return {N: np.stack(v) for N, v in per.items()}

    for what, nops in (("apply", 9),) + ((("advect", 1), ("biased", 3)) if g in (4, 6) else ()):
        got, want = call(what, lib.CFD_TC_BF16_EXACT, nops), call(what, lib.CFD_FP64_BANDED, nops)
        for N in got:
            for q in range(nf):
                for i in range(nops):
                    e = rel_max(got[N][:, q, i], want[N][:, q, i])
                    assert e < tol, (what, N, q, i, e)


def test_dissipation_of_tiny_fields(lib):
    """Fields near 2^-130: the FP32 dissipation sums are subnormal floats there and keep what those hold (2^-19 of
    the fields), so the step is the ordinary one scaled, to a hundredth of what the dissipation contributes."""
    import torch
    from oracle import timestep as T
    N, g, S = 16, 4, 2.0 ** -130
    mesh = W.periodic_box_mesh(2, 2, 2, N, g)
    E = N + 2 * g
    flat = W.rng(41).uniform(-1, 1, (8, 2, E ** 3))
    s = lib.cfd_scheme_create(desc("Q13_1_d1"), desc("Q13_1_d2"))
    B = lib.cfd_blocks_bind(s, mesh.n, mesh.dx, mesh.neighbors, g, lib.CFD_F64)
    dev, I = torch.device("cuda", 0), slice(g, g + N)

    def step(scale, sigma):
        u = [torch.from_numpy(flat[:, q].reshape(-1) * scale).to(dev) for q in range(2)]
        work = torch.empty(lib.cfd_wave_lsrk_workspace(B, lib.CFD_TC_BF16_EXACT, 0), dtype=torch.uint8, device=dev)
        lib.cfd_wave_lsrk_step(B, u[0], u[1], 0.1 * mesh.dx.min(), T.lsrk2s_rk4_float(), sigma, 4,
                               lib.CFD_TC_BF16_EXACT, 0, work)
        lib.cfd_sync_status(B)
        return np.stack([v.cpu().numpy().reshape(8, E, E, E)[:, I, I, I] for v in u]) / scale

    tiny, ordinary, without = step(S, 0.4), step(1.0, 0.4), step(1.0, 0.0)
    for q in range(2):
        effect = np.abs(ordinary[q] - without[q]).max()
        assert effect > 0
        assert np.abs(tiny[q] - ordinary[q]).max() < 1e-2 * effect, q
