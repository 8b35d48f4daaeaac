"""Different handles in different host threads: each gives what it gives alone, bit for bit.

The launch shapes of two batches (block sizes of the reconstruction and flux kernels, as the
autotuner may choose them) and the shared memory of two meshes' GMRES (several cells per
thread: it grows with the mesh) differ on purpose.
"""
import os
import subprocess
import sys
import threading
import time

import pytest

import handle_shim
import paper_2304_09485_gb300 as H
from paper_2304_09485_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def shim(cuda, tmp_path_factory):
    return handle_shim.load(tmp_path_factory.mktemp("shim"))


def together(jobs):
    """Runs the jobs in a thread each, started together; raises what a job raised."""
    gate, errors = threading.Barrier(len(jobs)), []

    def body(job):
        try:
            gate.wait()
            job()
        except Exception as e:      # noqa: BLE001
            errors.append(e)
    threads = [threading.Thread(target=body, args=(j,)) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    if errors:
        raise errors[0]


@pytest.mark.parametrize("scheme", [0, 1], ids=["weno", "hweno"])
def test_batches_of_different_shapes(shim, scheme):
    import torch
    m, cond = I.cavity_mesh(3), I.cavity_conditions()
    Q, G = I.smooth_state(m, amp=0.05, base=(1.0, 0.1, 0.05, -0.03, cond["p_inf"]))
    p = H.hgks_default_params(scheme=scheme, Pr=0.72, krylov_dim=2, restarts=1, **cond)
    hm = H.hgks_mesh_create(m, scheme_mask=1 << scheme)
    Qd, Gd = hm.to_internal(Q), hm.to_internal(G)
    batches, want = [], []
    for shape in (64, 256):
        b = H.hgks_batch_create([hm], [p])
        shim.hx_batch_shape(b.handle, shape, shape)
        H.hgks_batch_set_state(b, 0, Qd, Gd if scheme else None)
        H.hgks_batch_residual(b)
        R = torch.empty_like(Qd)
        H.hgks_batch_get_state(b, 0, R=R)
        torch.cuda.synchronize()
        batches.append(b)
        want.append(R)

    def job(k):
        stream = torch.cuda.Stream()
        R = torch.empty_like(Qd)
        with torch.cuda.stream(stream):
            for _ in range(1500):
                H.hgks_batch_residual(batches[k])
            H.hgks_batch_get_state(batches[k], 0, R=R)
            stream.synchronize()
        assert torch.equal(R, want[k])
    together([lambda k=k: job(k) for k in range(2)])


LIMITS = """
import handle_shim, sys
import paper_2304_09485_gb300 as H
from paper_2304_09485_gb300 import inputs as I
shim = handle_shim.load(sys.argv[1])
for make, cond in ((lambda: I.cavity_mesh(3), I.cavity_conditions()), (lambda: I.hex_cavity_mesh(4), I.cavity_conditions())):
    m = make()
    hm = H.hgks_mesh_create(m, scheme_mask=3)
    Q, G = (hm.to_internal(a) for a in I.smooth_state(m, amp=0.05, base=(1.0, 0.1, 0.05, -0.03, cond["p_inf"])))
    for scheme in (0, 1):
        for shape in (64, 128, 256):
            b = H.hgks_batch_create([hm], [H.hgks_default_params(scheme=scheme, Pr=0.72, **cond)])
            shim.hx_batch_shape(b.handle, shape, shape)
            H.hgks_batch_set_state(b, 0, Q, G if scheme else None)
            H.hgks_batch_residual(b)
cond = I.sphere_conditions(0.3)
for n, layers in ((2, 4), (6, 8), (9, 21), (13, 26)):
    m = I.sphere_mesh(n, layers, stretch=I.sphere_stretch(layers))
    hm = H.hgks_mesh_create(m, scheme_mask=1)
    H.hgks_gmres_step(hm, H.hgks_default_params(krylov_dim=2, restarts=1, **cond), hm.to_internal(I.state_from_conditions(m.n_tet, cond)))
H.hgks_sync()
"""


def test_a_kernels_limit_has_one_value(cuda, tmp_path):
    """Dynamic shared memory is allowed per kernel and process: whatever handle and shape a call
    comes with, it sets the same value."""
    log = str(tmp_path / "limits")
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    env = dict(os.environ, LD_PRELOAD=handle_shim.limit_recorder(tmp_path), HGKS_LIMIT_LOG=log,
               PYTHONPATH=os.pathsep.join([root, os.path.join(root, "tests")]))
    subprocess.run([sys.executable, "-c", LIMITS, str(tmp_path)], check=True, env=env)
    seen = {}
    for line in open(log):
        kernel, value = line.split()
        seen.setdefault(kernel, set()).add(int(value))
    # k_recon and k_flux: two cell kinds in a batch (compact and not: two of each on hexahedra, and
    # one k_recon on tetrahedra) and tetrahedra alone; the one-launch GMRES in three forms at least
    assert len(seen) >= 7 + 2 + 3, seen
    assert all(len(v) == 1 for v in seen.values()), seen


def test_meshes_of_different_sizes(cuda):
    """A step captures its launches anew when its parameters change: every step does here."""
    import torch
    cond = I.sphere_conditions(0.3)
    meshes = [I.sphere_mesh(n, layers, stretch=I.sphere_stretch(layers)) for n, layers in ((9, 21), (13, 26))]
    handles = [H.hgks_mesh_create(m, scheme_mask=1) for m in meshes]
    starts = [h.to_internal(I.state_from_conditions(m.n_tet, cond)) for h, m in zip(handles, meshes)]
    steps = 150

    def run(k):
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            Q, out = torch.empty_like(starts[k]), torch.empty(steps, dtype=torch.float64, device="cuda")
            for i in range(steps):
                Q.copy_(starts[k])
                p = H.hgks_default_params(krylov_dim=2, restarts=1, jacobi_sweeps=1, **{**cond, "cfl": 5.0 + 0.02 * i})
                H.hgks_gmres_step(handles[k], p, Q, None)
                out[i] = (Q * torch.arange(1, Q.numel() + 1, dtype=torch.float64, device="cuda").view_as(Q).sin()).sum()
            stream.synchronize()
        return out
    alone = [run(k) for k in range(2)]
    got = [None, None]

    def job(k):
        got[k] = run(k)
    together([lambda k=k: job(k) for k in range(2)])
    for k in range(2):
        assert torch.equal(got[k], alone[k]), (got[k] != alone[k]).nonzero().flatten().tolist()[:10]


def test_small_meshes_on_their_own_streams_overlap(cuda):
    """A one-launch GMRES takes 41 SMs for 1,296 cells, so three of them run side by side: eight
    threads' steps must end in less than 0.6 of the time that they take one after the other."""
    import torch
    m, cond = I.cavity_mesh(6), I.cavity_conditions(0.15, 100.0)
    p = H.hgks_default_params(scheme=0, Pr=0.72, **cond)
    handles = [H.hgks_mesh_create(m, scheme_mask=1) for _ in range(8)]
    Q0 = handles[0].to_internal(I.smooth_state(m, amp=0.02, base=(1.0, 0.05, 0.03, -0.02, cond["p_inf"]))[0])
    states, streams = [Q0.clone() for _ in handles], [torch.cuda.Stream() for _ in handles]
    torch.cuda.synchronize()

    def job(k, steps):
        with torch.cuda.stream(streams[k]):
            for _ in range(steps):
                H.hgks_gmres_step(handles[k], p, states[k])
    together([lambda k=k: job(k, 3) for k in range(8)])
    t0 = time.perf_counter()
    for k in range(8):
        job(k, 40)
    t1 = time.perf_counter()
    together([lambda k=k: job(k, 40) for k in range(8)])
    t2 = time.perf_counter()
    assert all(torch.equal(s, states[0]) for s in states)
    assert t2 - t1 < 0.6 * (t1 - t0), (t1 - t0, t2 - t1)
