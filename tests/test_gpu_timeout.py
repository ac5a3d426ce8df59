"""The device-side timeout path of the tensor-core kernel, exercised without a fault or a hang.

Every wait inside the kernel's main loop is bounded; when one runs out the kernel latches
CFD_ERR_TIMEOUT in the handle's status word, drains its own TMA copies and MMAs (with the
long default limit) and frees its tensor memory.  The test hook cfd_debug_set_wait_limit
makes the limit a few cycles, so that the first wait of every role gives up at once: nothing
hangs, the host sees the status, and the next call with the default limit is correct.
"""
import numpy as np
import pytest

from oracle import cfd as C
from paper_2302_14858_gb300 import workloads as W
from tests.helpers import OPS, desc, oracle_sch, rel_max

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    from paper_2302_14858_gb300 import build
    build.build()
    from paper_2302_14858_gb300 import cfd
    return cfd


@pytest.mark.parametrize("n_iter", [0, 1])
def test_wait_limit_runs_out_then_next_call_is_correct(lib, n_iter):
    import torch
    NM, N, g = 64, 32, 4
    dx = 2 * np.pi / NM
    x = (np.arange(NM) + 0.5) * dx
    Z, Y, X = np.meshgrid(x, x, x, indexing="ij")
    f = W.sine_sum(W.rng(61), 8, 1, 12)
    ext = C.ghost_fill_3d(f(X, Y, Z), N, g)
    mesh = W.uniform_mesh(NM, N, g)
    s = lib.cfd_scheme_create(desc("Q13_1_d1"), desc("Q13_1_d2"))
    B = lib.cfd_blocks_bind(s, mesh.n, mesh.dx, mesh.neighbors, g, lib.CFD_F64)
    dev = torch.device("cuda", 0)
    fields = torch.from_numpy(ext.reshape(-1).copy()).to(dev)
    out = torch.empty(mesh.nblocks * 9 * N ** 3, dtype=torch.float64, device=dev)
    ws = lib.cfd_apply_workspace(B, 1, lib.CFD_OP_ALL, lib.CFD_TC_BF16_EXACT, n_iter)
    work = torch.empty(max(ws, 256), dtype=torch.uint8, device=dev)
    lib.cfd_debug_set_wait_limit(4)
    try:
        lib.cfd_apply(B, fields, 1, lib.CFD_OP_ALL, lib.CFD_TC_BF16_EXACT, n_iter, out, work)
        with pytest.raises(lib.CfdError) as e:
            lib.cfd_sync_status(B)
        assert e.value.status == lib.CFD_ERR_TIMEOUT
    finally:
        lib.cfd_debug_set_wait_limit(0)
    lib.cfd_sync_status(B)                      # cleared by the read above
    out.fill_(float("nan"))
    lib.cfd_apply(B, fields, 1, lib.CFD_OP_ALL, lib.CFD_TC_BF16_EXACT, n_iter, out, work)
    lib.cfd_sync_status(B)
    got = out.cpu().numpy().reshape(mesh.nblocks, 9, N, N, N)
    ref = C.apply_uniform(ext, oracle_sch("Q13_1_d1"), oracle_sch("Q13_1_d2"), (dx, dx, dx), N, g, OPS, n_iter)
    for i, op in enumerate(OPS):
        assert rel_max(got[:, i], ref[op].reshape(mesh.nblocks, N, N, N)) < 1e-7, op


EARLY = r"""
// Lets the next chained launch start at once, then runs on for `cycles` clock cycles.
__global__ void early(long long cycles) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const long long t0 = clock64();
  while (clock64() - t0 < cycles) {}
}
extern "C" int early_launch(long long cycles, void *stream) {
  early<<<1, 32, 0, (cudaStream_t)stream>>>(cycles);
  return (int)cudaGetLastError();
}
"""


@pytest.mark.parametrize("n_iter", [0, 1])
def test_wait_limit_does_not_count_the_launch_before(lib, tmp_path, n_iter):
    """A caller's kernel that triggers its dependents early and runs on for ten times the wait limit: the
    chained launch behind it starts its waits when that kernel has ended, so none runs out."""
    import ctypes
    import subprocess

    import torch
    from paper_2302_14858_gb300 import build
    src, so = tmp_path / "early.cu", tmp_path / "early.so"
    src.write_text(EARLY)
    subprocess.run([build.nvcc()] + build.ARCH + ["-shared", "-Xcompiler", "-fPIC", "-o", str(so), str(src)], check=True)
    early = ctypes.CDLL(str(so)).early_launch
    early.argtypes = [ctypes.c_longlong, ctypes.c_void_p]
    N, g = 32, 4
    mesh = W.periodic_box_mesh(2, 1, 1, N, g)
    s = lib.cfd_scheme_create(desc("Q13_1_d1"), desc("Q13_1_d2"))
    B = lib.cfd_blocks_bind(s, mesh.n, mesh.dx, mesh.neighbors, g, lib.CFD_F64)
    dev = torch.device("cuda", 0)
    fields = torch.from_numpy(W.rng(7).uniform(-1, 1, 2 * (N + 2 * g) ** 3)).to(dev)
    mask = lib.op_mask(("dx", "dyy"))
    outs = [torch.empty(2 * 2 * N ** 3, dtype=torch.float64, device=dev) for _ in range(2)]
    work = torch.empty(max(lib.cfd_apply_workspace(B, 1, mask, lib.CFD_TC_BF16_EXACT, n_iter), 256),
                       dtype=torch.uint8, device=dev)
    lib.cfd_apply(B, fields, 1, mask, lib.CFD_TC_BF16_EXACT, n_iter, outs[0], work)
    lib.cfd_sync_status(B)
    limit = 2_000_000                           # about 1 ms; the launches themselves take ~10 us
    lib.cfd_debug_set_wait_limit(limit)
    try:
        assert early(10 * limit, torch.cuda.current_stream().cuda_stream) == 0
        lib.cfd_apply(B, fields, 1, mask, lib.CFD_TC_BF16_EXACT, n_iter, outs[1], work)
        lib.cfd_sync_status(B)
    finally:
        lib.cfd_debug_set_wait_limit(0)
    assert torch.equal(outs[0], outs[1])
