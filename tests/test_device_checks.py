"""What the C ABI cannot reach of the device code, through a small library
compiled from it: waits that run out, tables that are full."""

import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2411_11244_gb300 import synth

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


def _compile(tmp, name, *defines):
    from paper_2411_11244_gb300 import build as B
    out = os.path.join(tmp, name + ".so")
    src = [os.path.join(HERE, "native", "device_checks.cu"), os.path.join(B.CSRC, "gd_build.cu"),
           os.path.join(B.CSRC, "gd_point.cu")]
    cmd = [B.nvcc(), *B.FLAGS, *B.ARCH, *defines, "-I", B.CSRC, "-shared", "-o", out, *src]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    lib = ctypes.CDLL(out)
    lib.check_block.restype = ctypes.c_void_p
    return lib


@pytest.fixture(scope="module")
def G():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2411_11244_gb300 import gdist
    return gdist


@pytest.fixture(scope="module")
def checks(tmp_path_factory):
    return _compile(str(tmp_path_factory.mktemp("native")), "checks")


@pytest.mark.parametrize("n", [1025, 100_003, 300_001])
def test_sort_that_gives_up_writes_nothing(checks, n):
    """A tile of the first pass never publishes: the waits for it run out, the
    passes that follow leave their buffers alone (the pairs that the first pass
    did not write would be placed beyond them), and the error word is set.  The
    waits end after the limit that the sort was given: 2 ms here, and far less than
    the 2 s of a context's default with the launches around them."""
    rng = np.random.default_rng(n)
    keys = rng.integers(0, 1 << 63, n, dtype=np.uint64)
    p = keys.ctypes.data_as(ctypes.c_void_p)
    ms = ctypes.c_double()
    assert checks.check_sort_gives_up(p, ctypes.c_longlong(n), 4, ctypes.c_ulonglong(2_000_000), ctypes.byref(ms)) == 0
    assert 2.0 <= ms.value < 500.0


def test_graph_after_a_batch_that_moves_the_refit_table(G, checks):
    """The queues are at their limit, so a batch against a deep tree moves only
    the table of refit roots (64 x 2^11 entries).  A graph made before is made
    again by its next launch: it gives the plain call's answer, and what lies
    where the table was stays as it is."""
    torch = pytest.importorskip("torch")
    ctx = G.gd_ctx_create(0)
    try:
        cap = 1 << 20
        G.gd_ctx_set_tunables(ctx, front_capacity=cap, leaf_capacity=cap, cand_capacity=1 << 18, max_capacity=cap,
                              batch_budget=cap >> 7)

        def mesh(m):
            h = G.gd_mesh_create(ctx, *m)
            G.gd_bvh_build(h, ctx=ctx)
            return h

        a, small, deep = (mesh(m) for m in (synth.torus(1.0, 0.3, 40, 40), synth.geosphere(12, 0.5),
                                            synth.geosphere(163, 0.5)))
        assert G.gd_mesh_info(deep)[0] == 19
        I = synth.identity_xform()
        xs = [synth.xform(np.eye(3), (2.0 + 0.01 * i, 0.1, 0.2)) for i in range(64)]
        G.gd_batch_query(ctx, G.make_queries([(a, small, I, x, G.GD_MIN) for x in xs]))
        ref = G.gd_min_distance(ctx, a, small, I, xs[5])
        dxa = torch.tensor(I, dtype=torch.float64, device="cuda")
        dxb = torch.tensor(xs[5], dtype=torch.float64, device="cuda")
        out = torch.zeros(10, dtype=torch.float64, device="cuda")
        g = G.gd_graph_create(ctx, a, small, G.GD_MIN, dxa.data_ptr(), dxb.data_ptr(), out.data_ptr())
        G.gd_batch_query(ctx, G.make_queries([(a, deep, I, x, G.GD_MIN) for x in xs]))
        size = 4 << 16  # the table before the batch
        blocks = [checks.check_block(ctypes.c_size_t(size), 0x5a) for _ in range(64)]
        assert all(blocks)
        torch.cuda.synchronize()
        G.gd_graph_launch(g, None, ctx)
        torch.cuda.synchronize()
        r = G.gd_result.from_buffer_copy(out.cpu().numpy().tobytes())
        kept = [checks.check_block_kept(ctypes.c_void_p(b), ctypes.c_size_t(size), 0x5a) for b in blocks]
        assert kept == [1] * 64
        assert (r.status, r.d, r.tri_a, r.tri_b) == (0, ref.d, ref.tri_a, ref.tri_b)
        G.gd_graph_destroy(g)
        for h in (a, small, deep):
            G.gd_mesh_destroy(h)
    finally:
        G.gd_ctx_destroy(ctx)


@pytest.mark.parametrize("room", [None, (3, 9), (2, 64), (64, 2)])
def test_points_with_shared_walks(G, tmp_path, checks, room):
    """Points around the centre of a sphere, whose walks meet all of it: warps give
    parts of them away, as the counters show, also when there is too little room for
    the points that want to share or for their gifts, and in a second call over the
    first one's records.  Every answer is that of the same point in a call by itself
    (and of gd_point_distance for all of them)."""
    lib = checks
    if room:
        lib = _compile(str(tmp_path), "room", f"-DGD_POINT_SLOTS={room[0]}u", f"-DGD_POINT_SHARES={room[1]}u")
    v, t = synth.geosphere(64, 1.0, 1e-4, 3)
    n = 200
    pts = np.random.default_rng(9).normal(0.0, 1e-3, (n, 3))
    out = (G.gd_point_result * (2 * n))()
    c = [ctypes.c_ulonglong() for _ in range(3)]
    p = [a.ctypes.data_as(ctypes.c_void_p) for a in (v, t, pts)]
    assert lib.check_points(p[0], ctypes.c_longlong(len(v)), p[1], ctypes.c_longlong(len(t)), p[2],
                            ctypes.c_longlong(n), out, *map(ctypes.byref, c)) == 0
    slots, gifts, parts = (x.value for x in c)
    if room is None:
        assert slots > 0 and gifts > slots and parts > 0
    else:
        assert slots > room[0] or gifts > room[1]
    ctx = G.gd_ctx_create(0)
    try:
        h = G.gd_mesh_create(ctx, v, t)
        G.gd_bvh_build(h, ctx=ctx)
        ref = G.gd_point_distance(ctx, h, synth.identity_xform(), pts)
        for i in (0, 7, n - 1):
            one = G.gd_point_distance(ctx, h, synth.identity_xform(), pts[i:i + 1])
            assert one.tobytes() == ref[i:i + 1].tobytes()
        G.gd_mesh_destroy(h)
    finally:
        G.gd_ctx_destroy(ctx)
    assert (ref["status"] == 0).all()
    got = np.frombuffer(out, dtype=ref.dtype)
    for f in ("d", "tri", "p", "status"):
        assert np.array_equal(got[f][:n], ref[f]) and np.array_equal(got[f][n:], ref[f])
