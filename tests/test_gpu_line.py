"""The FP64 pencil solves on meshes that the uniform parity tests do not reach: spacing that differs
between blocks of one size, stencils that are antisymmetric only to rounding, blocks that are cyclic
along an axis beside blocks that are not, several iterations with FP32 fields.  Tolerance 1e-12 of the
largest output for FP64 (the parity tests' own), 2e-6 for FP32 fields.
"""
import numpy as np
import pytest

from paper_2302_14858_gb300 import workloads as W
from tests.helpers import desc, rel_max

pytestmark = pytest.mark.gpu
OPS = ("dx", "dy", "dz", "dxx", "dyy", "dzz", "dxy", "dxz", "dyz")


@pytest.fixture(scope="module")
def lib():
    from paper_2302_14858_gb300 import build
    build.build()
    from paper_2302_14858_gb300 import cfd
    return cfd


def run(lib, first, second, n, dx, nbr, g, flat, nf, ops, n_iter, f32=False):
    import torch
    s = lib.cfd_scheme_create(first, second)
    B = lib.cfd_blocks_bind(s, n, dx, nbr, g, lib.CFD_F32 if f32 else lib.CFD_F64)
    dev = torch.device("cuda", 0)
    f = torch.from_numpy(np.ascontiguousarray(flat, np.float32 if f32 else np.float64)).to(dev)
    mask = lib.op_mask(ops)
    nint = sum(int(v) ** 3 for v in n)
    out = torch.full((nint * nf * len(ops),), float("nan"), dtype=f.dtype, device=dev)
    ws = lib.cfd_apply_workspace(B, nf, mask, lib.CFD_FP64_BANDED, n_iter)
    work = torch.empty(max(ws, 256), dtype=torch.uint8, device=dev)
    lib.cfd_apply(B, f, nf, mask, lib.CFD_FP64_BANDED, n_iter, out, work)
    lib.cfd_sync_status(B)
    N = int(n[0])
    return out.cpu().numpy().astype(np.float64).reshape(len(n), nf, len(ops), N, N, N)


def field(mesh, nf, seed, f32=False):
    r = W.rng(seed)
    L = [(mesh.origin[:, a].max() + mesh.n[0]) * mesh.dx[0, a] for a in range(3)]
    fs = []
    for _ in range(nf):
        s = W.sine_sum(r, 6, 1, 3)
        s.k = 2 * np.pi * s.k / np.asarray(L)
        fs.append(s)
    return W.pack(W.sample(mesh, fs, np.float32 if f32 else np.float64))


@pytest.mark.parametrize("N", [8, 16, 32])
def test_spacing_that_differs_between_blocks(lib, N):
    mesh = W.periodic_box_mesh(2, 3, 2, N, 4)
    flat = field(mesh, 2, 5 + N)
    dx = np.array(mesh.dx)
    dx *= (1.0 + 0.25 * np.arange(len(dx)))[:, None] * np.array([1.0, 0.5, 2.0])
    got = run(lib, desc("Q13_1_d1"), desc("Q13_1_d2"), mesh.n, dx, mesh.neighbors, 4, flat, 2, OPS, 0)
    one = run(lib, desc("Q13_1_d1"), desc("Q13_1_d2"), mesh.n, np.ones_like(dx), mesh.neighbors, 4, flat, 2, OPS, 0)
    for i, op in enumerate(OPS):  # closed blocks: every block's operator scales with its own spacing
        h = np.prod([dx[:, "xyz".index(c)] for c in op[1:]], axis=0) if len(op) > 2 else dx[:, "xyz".index(op[1])]
        assert rel_max(got[:, :, i] * h[:, None, None, None, None], one[:, :, i]) < 1e-12, op


@pytest.mark.parametrize("n_iter", [0, 1, 2])
def test_stencils_antisymmetric_to_rounding_only(lib, n_iter):
    mesh = W.periodic_box_mesh(3, 2, 1, 16, 4)
    flat = field(mesh, 1, 9)
    a, b = desc("Q13_1_d1"), desc("Q13_1_d2")
    got0 = run(lib, a, b, mesh.n, mesh.dx, mesh.neighbors, 4, flat, 1, OPS, n_iter)
    a2 = dict(a, rhs=list(a["rhs"]))
    a2["rhs"][0] *= 1.0 + 4e-15
    got1 = run(lib, a2, b, mesh.n, mesh.dx, mesh.neighbors, 4, flat, 1, OPS, n_iter)
    for i, op in enumerate(OPS):
        assert rel_max(got1[:, :, i], got0[:, :, i]) < 1e-12, op


@pytest.mark.parametrize("N,n_iter", [(8, 0), (8, 2), (16, 1), (32, 1)])
def test_cyclic_blocks_beside_others(lib, N, n_iter):
    """Block 0 is a periodic mesh of its own; blocks 1 and 2 are a ring along x (cyclic along y, z)."""
    g = 4
    single, ring = W.periodic_box_mesh(1, 1, 1, N, g), W.periodic_box_mesh(2, 1, 1, N, g)
    f0, f1 = field(single, 1, 3), field(ring, 1, 4)
    d = (desc("Q13_1_d1"), desc("Q13_1_d2"))
    dx = np.full((3, 3), 0.1)
    nbr = np.concatenate([np.array(single.neighbors), np.array(ring.neighbors) + 1]).astype(np.int32)
    got = run(lib, *d, [N] * 3, dx, nbr, g, np.concatenate([f0, f1]), 1, OPS, n_iter)
    w0 = run(lib, *d, [N], dx[:1], single.neighbors, g, f0, 1, OPS, n_iter)
    w1 = run(lib, *d, [N] * 2, dx[:2], ring.neighbors, g, f1, 1, OPS, n_iter)
    want = np.concatenate([w0, w1])
    for i, op in enumerate(OPS):
        assert rel_max(got[:, :, i], want[:, :, i]) < 1e-13, op


@pytest.mark.parametrize("ops,n_iter", [(OPS, 2), (("dxy",), 1), (("dx", "dyz"), 0), (("dzz", "dxz", "dyz"), 2)])
def test_op_subsets_and_fp32_agree_with_fp64(lib, ops, n_iter):
    """Mixed ops with and without their inner derivative among the outputs, FP64 and FP32 fields."""
    mesh = W.periodic_box_mesh(2, 2, 3, 16, 4)
    flat = field(mesh, 2, 21, f32=True)
    d = (desc("Q13_1_d1"), desc("Q13_1_d2"))
    full = run(lib, *d, mesh.n, mesh.dx, mesh.neighbors, 4, flat, 2, OPS, n_iter)
    some = run(lib, *d, mesh.n, mesh.dx, mesh.neighbors, 4, flat, 2, ops, n_iter)
    f32 = run(lib, *d, mesh.n, mesh.dx, mesh.neighbors, 4, flat, 2, ops, n_iter, f32=True)
    for i, op in enumerate(ops):
        want = full[:, :, OPS.index(op)]
        assert rel_max(some[:, :, i], want) < 1e-13, op
        assert rel_max(f32[:, :, i], want) < 2e-6, op


@pytest.mark.parametrize("N,g,wide", [(32, 6, 2), (32, 6, 1), (16, 6, 2), (32, 8, 2)])
def test_a_wider_stencil_of_the_other_degree_changes_nothing(lib, N, g, wide):
    """A scheme whose other degree has the widest closure there is (half-width 6): the requested degree's
    solves are the same bits as with the ordinary scheme, and the call is accepted as such."""
    mesh = W.periodic_box_mesh(2, 1, 1, N, g)
    flat = field(mesh, 1, 31 + N)
    d = [desc("Q13_1_d1"), desc("Q13_1_d2")]
    ops = ("dx", "dy", "dz", "dxy") if wide == 2 else ("dxx", "dyy", "dzz")
    want = run(lib, *d, mesh.n, mesh.dx, mesh.neighbors, g, flat, 1, ops, 1)
    c = d[wide - 1]["closure"]
    pad = [0.0] * ((13 - len(c)) // 2)
    d[wide - 1] = dict(d[wide - 1], closure=pad + list(c) + pad)
    got = run(lib, *d, mesh.n, mesh.dx, mesh.neighbors, g, flat, 1, ops, 1)
    assert np.array_equal(got, want)


@pytest.mark.parametrize("N,ops", [(8, ("dx", "dyy", "dz")), (16, ("dxx", "dy", "dzz")), (32, ("dx", "dz"))])
def test_fp32_fields_are_widened_exactly(lib, N, ops):
    """FP32 fields of every kind (normal, subnormal, zeros of either sign, the largest; one block with a NaN and
    an infinity) give the FP32 rounding of what the same values give as FP64 fields."""
    mesh = W.periodic_box_mesh(2, 2, 1, N, 4)
    E = N + 8
    r = W.rng(70 + N)
    f = r.uniform(-1, 1, (4, 1, E ** 3)) * 2.0 ** r.integers(-12, 12, (4, 1, E ** 3))
    f[1] *= 2.0 ** -140                               # subnormal in FP32, many to zero
    f[2, 0, ::3] = np.where(r.uniform(size=len(f[2, 0, ::3])) < 0.5, -0.0, 3e38)
    f[3, 0, E ** 3 // 2] = np.nan
    f[3, 0, E ** 3 // 2 + 5] = np.inf
    flat = f.astype(np.float32).reshape(-1)
    d = (desc("Q13_1_d1"), desc("Q13_1_d2"))
    dx = np.full((4, 3), 0.125)
    with np.errstate(over="ignore", invalid="ignore"):
        want = run(lib, *d, mesh.n, dx, mesh.neighbors, 4, flat.astype(np.float64), 1, ops, 0).astype(np.float32)
    got = run(lib, *d, mesh.n, dx, mesh.neighbors, 4, flat, 1, ops, 0, f32=True).astype(np.float32)
    assert np.array_equal(got, want, equal_nan=True)
