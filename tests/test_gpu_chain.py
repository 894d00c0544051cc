"""GPU tests of the Newton-Schulz chain: one launch that runs every phase of
every iteration, its tiles ordered by counters in global memory (Section 2's
iteration on the tensor cores).

The sizes are the edges of its choices: matrices inside one tile and just past
one, 128- and 256-column tiles (the switch is at one 256 x 256 APPLY tile per
CTA pair, 76 of them), Gram tiles whole and split along K, more shapes than one
launch takes (eight), and the stable-rank mask, whose tile lists are compacted
on the device."""

import numpy as np
import pytest

import oracle as O
from paper_2605_19811_gb300 import synth
from tests.lm_testutil import bits, host_tensor, ns_closed_form_rows, rel_fro, stored_values, tall

pytestmark = pytest.mark.gpu

QUINTIC = O.NS_QUINTIC


def _msign(xh, precision, steps=5):
    import torch
    from paper_2605_19811_gb300 import lionmuon as L
    out = torch.empty(xh.shape, dtype=torch.float32, device="cuda")
    L.msign_ns(xh.cuda(), out, steps, *QUINTIC, eps=1e-7, precision=precision)
    return stored_values(out)


# inside one tile; one past 128, 256; 384 = 1.5 tiles; a long Gram split into
# parts; 72 and 90 APPLY tiles of 256 x 256 (narrow and full-width tiles)
@pytest.mark.parametrize("shape", [(128, 256), (129, 257), (257, 255), (384, 384), (640, 12800), (12800, 250),
                                   (2000, 2100), (2100, 2400)])
@pytest.mark.parametrize("precision,dtype,tol", [(1, "bf16", 2e-2), (2, "f32", 2e-5)])
def test_msign_at_tile_edges(shape, precision, dtype, tol):
    xh = host_tensor(synth.draw_matrix(shape, seed=shape[0]), dtype)
    got = _msign(xh, precision)
    want = ns_closed_form_rows(stored_values(xh), 5, *QUINTIC, 1e-7)
    assert rel_fro(tall(got), want) <= tol


def _steps(shapes, profile, steps=3, dtype="bf16", **cfg):
    import torch
    from paper_2605_19811_gb300 import lionmuon as L
    params = [host_tensor(w, dtype).cuda() for w in synth.init_weights(shapes, seed=1)]
    opt = L.LionMuon(params, **cfg)
    if dtype == "f32" and cfg["ns_precision"] == 0:
        assert opt.ns_path() == L.LM_NS_F32_TC
    opt.profile(profile)
    for t in range(steps):
        opt.step([host_tensor(x, dtype).cuda() for x in synth.draw_grads(shapes, "student_t", seed=0, step=t)], t)
    torch.cuda.synchronize()
    assert opt.status() == 0
    out = [bits(p) for p in params] + [bits(opt.momentum(i)) for i in range(len(params))]
    opt.close()
    return out


# nine shapes: two launches; a 20000-long Gram split next to short ones; tables
# whose last iteration folds a and whose last does not; a wide set (256-column
# tiles) and a small one (128)
NINE = [(64 * k, 64 * k + 128) for k in range(1, 10)]
CASES = [(NINE, {}), ([(768, 768), (20000, 768), (768, 2304), (768,)], {}),
         ([(512, 640), (640, 512)], dict(ns_coeffs=((8.4, -25.0, 18.0), (4.1, -3.1, 0.6), (1.5, -0.5, 0.0)))),
         ([(768, 3072)] * 4, dict(ns_coeffs=((1.5, -0.5, 0.0), (3.4445, -4.775, 2.0315)))),
         ([(512, 1024), (1024, 512)] * 3, dict(schedule=1, srank_alpha=0.02))]


# the same kinds for the full-fp32 mode with register sums (every matrix wide
# enough for it): nine shapes, a long Gram split along K next to short matrices,
# tables with and without a cubic, the mask
WIDE_CASES = [([(320 + 32 * k, 448 + 32 * k) for k in range(9)], {}),
              ([(768, 768), (20000, 768), (768, 2304), (768,)], {}),
              ([(512, 640), (640, 512)], dict(ns_coeffs=((8.4, -25.0, 18.0), (4.1, -3.1, 0.6), (1.5, -0.5, 0.0)))),
              ([(512, 1024), (1024, 512)] * 3, dict(schedule=1, srank_alpha=0.02))]


@pytest.mark.parametrize("precision,dtype,shapes,cfg", [(p, d, *c) for p, d in ((1, "bf16"), (2, "f32")) for c in CASES] +
                         [(0, "f32", *c) for c in WIDE_CASES])
def test_one_launch_equals_one_launch_per_phase(shapes, cfg, precision, dtype):
    """With profiling on every phase has a launch of its own: the same tiles
    without the overlap of phases, so a missing dependency would show."""
    cfg = dict(period=1, **cfg) if "schedule" not in cfg else cfg
    a = _steps(shapes, False, dtype=dtype, ns_precision=precision, **cfg)
    b = _steps(shapes, True, dtype=dtype, ns_precision=precision, **cfg)
    for x, y in zip(a, b):
        np.testing.assert_array_equal(x, y)


# Element-wise kernels around the Newton-Schulz chain: row lengths that take
# units of 4, 2 and 1 elements and rows shorter than a vector, counts that are
# and are not multiples of 8 (the last elements), and a set small enough for
# short chunks next to one with whole chunks
@pytest.mark.parametrize("shape", [(37, 300), (300, 36), (64, 1202), (33, 301), (257, 5), (5, 3), (1201, 2), (2, 4099),
                                   (1000, 1301)])
@pytest.mark.parametrize("dtype,precision", [("bf16", 1), ("f32", 1), ("f32", 0), ("bf16", 0)])
def test_ragged_rows_step(shape, dtype, precision):
    """A Muon step against the storage-modelled oracle: momentum bit-exact,
    W <- W - eta (s NS(G_hat) + lambda W) within the NS tolerance."""
    import torch
    from paper_2605_19811_gb300 import lionmuon as L
    w0 = host_tensor(synth.init_weights([shape], seed=2)[0], dtype)
    g = host_tensor(synth.draw_matrix(shape, seed=7), dtype)
    p = w0.cuda()
    opt = L.LionMuon([p], period=1, eta_muon=0.02, weight_decay=0.1, ns_precision=precision)
    opt.step([g.cuda()], 0)
    torch.cuda.synchronize()
    assert opt.status() == 0
    m = (np.float32(1.0 - 0.99) * g.float().numpy()).astype(np.float32)
    np.testing.assert_array_equal(bits(opt.momentum(0)), m.view(np.uint32))
    gh = (np.float32(1.0 - 0.9) * g.float().numpy()).astype(np.float32).astype(np.float64)
    x = host_tensor(gh, "bf16") if precision == 1 else gh
    ns = ns_closed_form_rows(stored_values(x) if precision == 1 else x, 5, *QUINTIC, 1e-7)
    ns = ns if shape[0] >= shape[1] else ns.T
    upd = 0.02 * 0.2 * np.sqrt(max(shape)) * ns
    w = stored_values(w0)
    want = w - upd - 0.02 * 0.1 * w
    # the NS tolerance (2e-2 bf16, 1e-5 fp32), or 1.5 times what keeping X, A
    # and B in the path's storage type does to this input by itself (the
    # storage-modelled oracle; 2.1e-2 in bf16 on the 37 x 300 one)
    table = (QUINTIC,) * 5
    d = rel_fro(O.ns_polynomial_schedule_storage(gh, table, 1e-7, "bf16" if precision == 1 else "f32"),
                O.ns_polynomial_schedule(gh, table, 1e-7))
    tau = max(2e-2 if precision == 1 else 1e-5, 1.5 * d)
    # the NS tolerance of the update, and half a unit in the last place of W's
    # type per entry (2^-9 bf16, 2^-24 fp32)
    ulp = 2.0 ** -9 if dtype == "bf16" else 2.0 ** -24
    bound = tau * np.linalg.norm(upd) + 2 * ulp * np.linalg.norm(want)
    assert np.linalg.norm(stored_values(p) - want) <= bound
    opt.close()


# Full-fp32 mode around the choice of its path (with the quintic 256 rows, 512
# where the matrix is more than four times as long; 512 with another table),
# and on the CUDA cores: one 64-wide tile and just past it, tiles cut along K,
# 128-wide tiles
@pytest.mark.parametrize("shape", [(255, 600), (256, 600), (600, 256), (319, 700), (700, 320), (2, 64), (65, 64),
                                   (64, 5000), (250, 9000), (1000, 1024), (256, 1024), (1025, 256), (511, 2100),
                                   (2100, 512)])
def test_full_fp32_msign(shape):
    import torch
    from paper_2605_19811_gb300 import lionmuon as L
    from paper_2605_19811_gb300.ns_coeffs import polar_express
    xh = host_tensor(synth.draw_matrix(shape, seed=shape[0]), "f32")
    x = stored_values(xh)
    assert rel_fro(_msign(xh, 0), O.ns_polynomial(x, 5, *QUINTIC, 1e-7)) <= 1e-5
    if min(shape) >= 255:
        table = polar_express(5)
        out = torch.empty(shape, device="cuda")
        L.msign_ns_coeffs(xh.cuda(), out, table, precision=0)
        want = O.ns_polynomial_schedule(x, table, 1e-7)
        # 1e-5 for the quintic, scaled by how much more the table amplifies
        # fp32 storage on this input (the storage-modelled oracle; about 2)
        d = rel_fro(O.ns_polynomial_schedule_storage(x, table, 1e-7, "f32"), want)
        dq = rel_fro(O.ns_polynomial_schedule_storage(x, (QUINTIC,) * 5, 1e-7, "f32"), O.ns_polynomial(x, 5, *QUINTIC, 1e-7))
        assert rel_fro(stored_values(out), want) <= 1e-5 * max(1.0, d / dq)
    got = torch.empty(shape, device="cuda")
    L.msign_ns_noalloc(xh.cuda(), got, precision=0)   # CUDA cores at every size
    assert rel_fro(stored_values(got), O.ns_polynomial(x, 5, *QUINTIC, 1e-7)) <= 1e-5


def test_full_fp32_falls_back_without_the_workspace(monkeypatch):
    """No room for the three-piece workspace (injected): lm_create takes the
    CUDA-core path, with a workspace of its own size and the same step."""
    import torch
    from paper_2605_19811_gb300 import lionmuon as L
    shapes = [(320, 512), (512, 320)]
    g = [host_tensor(x, "f32").cuda() for x in synth.draw_grads(shapes, "student_t", seed=0, step=0)]
    out = []
    for fault in (None, "oom_f32tc"):
        if fault:
            monkeypatch.setenv("LM_FAULT", fault)
        params = [host_tensor(w, "f32").cuda() for w in synth.init_weights(shapes, seed=1)]
        opt = L.LionMuon(params, period=1, ns_precision=0)
        opt.step(g, 0)
        torch.cuda.synchronize()
        assert opt.status() == 0
        assert opt.ns_path() == (L.LM_F32 if fault else L.LM_NS_F32_TC)
        out.append(([stored_values(p) for p in params], opt.workspace_bytes()))
        opt.close()
    assert out[1][1] != out[0][1]
    for a, b in zip(out[0][0], out[1][0]):
        assert rel_fro(a, b) <= 1e-6   # the update is 3% of W, both NS within 1e-5


# 1-D parameters beside a bf16 matrix: of its dtype they take their Lion step in
# the momentum launch, of the other in a launch of their own; lengths around a
# vector of 8 and a chunk of 2048 elements, and many chunks
@pytest.mark.parametrize("n", [1, 7, 8, 2047, 2048, 2049, 70003])
@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_vectors_in_the_momentum_launch(n, dtype):
    """Bit-identical to the Lion kernel (with profiling on the vectors always
    have its launch)."""
    import torch
    from paper_2605_19811_gb300 import lionmuon as L
    shapes, dtypes = [(96, 200), (1, n), (1, 5)], ["bf16", dtype, "bf16"]
    got = []
    for profile in (False, True):
        params = [host_tensor(w, d).cuda() for w, d in zip(synth.init_weights(shapes, seed=3), dtypes)]
        opt = L.LionMuon(params, period=1, eta_lion=1e-3, weight_decay=0.1)
        opt.profile(profile)
        for t in range(3):
            gs = synth.draw_grads(shapes, "student_t", seed=4, step=t)
            opt.step([host_tensor(x, d).cuda() for x, d in zip(gs, dtypes)], t)
        torch.cuda.synchronize()
        assert opt.status() == 0
        got.append([bits(p) for p in params] + [bits(opt.momentum(i)) for i in range(3)])
    for x, y in zip(*got):
        np.testing.assert_array_equal(x, y)


def _device_step(shapes, profile, ranked=(), steps=1, **cfg):
    """Steps over bf16 sets too large to draw on the host; the matrices in
    ``ranked`` have a dominant direction in their gradients.  Returns the bits,
    the selection of the last step and its kernel launches."""
    import torch
    from paper_2605_19811_gb300 import lionmuon as L
    gen = torch.Generator(device="cuda")
    gen.manual_seed(5)

    def rand(s):
        return torch.randn(s, generator=gen, device="cuda")
    params = [(rand(s) * 0.02).bfloat16() for s in shapes]
    grads = [rand(s) for s in shapes]
    for i in ranked:
        grads[i] += 0.5 * rand(shapes[i][:1])[:, None] * rand(shapes[i][1:])[None, :]
    grads = [g.bfloat16() for g in grads]
    opt = L.LionMuon(params, **cfg)
    opt.profile(profile)
    for t in range(steps):
        n0 = L.kernel_launch_count()
        opt.step(grads, t)
        launches = L.kernel_launch_count() - n0
    torch.cuda.synchronize()
    assert opt.status() == 0
    out = [bits(x) for i in range(len(shapes)) for x in (params[i], opt.momentum(i))]
    took = opt.selection()[0]
    opt.close()
    return out, took, launches


@pytest.mark.parametrize("shapes,ranked", [
    ([(20000, 768), (768, 768), (768, 2304), (20000, 768)], (0, 1)),    # a light batch: Grams cut for the longest
    ([(16384, 2048), (2048, 2048), (16384, 2048)], (2,))])              # a heavy one: parts capped under the mask
def test_masked_lists_with_split_grams(shapes, ranked):
    """Selected and skipped matrices, both with Gram tiles split along K: one
    launch equals one launch per phase."""
    cfg = dict(schedule=1, srank_alpha=0.03, steps=3, ranked=ranked)
    a, took, _ = _device_step(shapes, False, **cfg)
    b, _, _ = _device_step(shapes, True, **cfg)
    assert took == [i in ranked for i in range(len(shapes))]
    for x, y in zip(a, b):
        np.testing.assert_array_equal(x, y)


def test_launch_per_phase_by_size_equals_one_launch():
    """A batch large enough for a launch per phase (nine 4096 x 4096: 4377 K
    blocks per CTA pair and iteration, from 4096), against the same tiles in
    one launch: under the stable-rank mask a batch always takes one, and at
    alpha = 1 every matrix is selected."""
    shapes = [(4096, 4096)] * 9
    a, _, na = _device_step(shapes, False, period=1)
    b, took, nb = _device_step(shapes, False, schedule=1, srank_alpha=1.0)
    assert all(took) and na - nb > 0, (na, nb)
    for x, y in zip(a, b):
        np.testing.assert_array_equal(x, y)


# long products, split along K, in the full-fp32 mode on either path
@pytest.mark.parametrize("shape", [(320, 20000), (512, 20000), (20000, 555)])
def test_full_fp32_msign_long(shape):
    xh = host_tensor(synth.draw_matrix(shape, seed=shape[0]), "f32")
    want = ns_closed_form_rows(stored_values(xh), 5, *QUINTIC, 1e-7)
    assert rel_fro(tall(_msign(xh, 0)), want) <= 1e-5


@pytest.mark.parametrize("shape,table", [((384, 15360), (QUINTIC,) * 5), ((480, 1440), (QUINTIC,) * 10),
                                         ((336, 504), "polar"), ((512, 768), "polar"), ((256, 1024), (QUINTIC,) * 5),
                                         ((1024, 1100), (QUINTIC,) * 10)])
def test_full_fp32_is_as_close_as_the_cuda_cores(shape, table, monkeypatch):
    """Whatever path LM_F32 takes, its direction is no further from fp64 than
    the CUDA cores' (the path it falls back to without the workspace), 10%
    allowed for the draw: the mean over inputs is below 1 where it takes the
    other one, 1.26 to 1.4 in the first three cases if it did."""
    import torch
    from paper_2605_19811_gb300 import lionmuon as L
    from paper_2605_19811_gb300.ns_coeffs import polar_express
    table = polar_express(5) if table == "polar" else table
    err = []
    x = host_tensor(synth.draw_matrix(shape, seed=shape[1]), "f32")
    want = O.ns_polynomial_schedule(stored_values(x), table, 1e-7)
    for fault in (None, "oom_f32tc"):
        if fault:
            monkeypatch.setenv("LM_FAULT", fault)
        w = torch.zeros(shape, device="cuda")
        opt = L.LionMuon([w], period=1, eta_muon=1.0, weight_decay=0.0, beta1=0.0, shape_scale=1.0, ns_precision=0,
                         ns_coeffs=table)
        opt.step([x.cuda()], 0)   # W = -sqrt(max(m, n)) NS(G)
        torch.cuda.synchronize()
        assert opt.status() == 0
        err.append(rel_fro(-stored_values(w) / max(shape) ** 0.5, want))
        opt.close()
    assert err[0] <= 1.1 * err[1], err


def test_three_piece_gram_parts_of_a_large_matrix():
    """A matrix whose Gram tiles come to more than 65535 parts of 128 columns
    (20480 x 20480: 3240 blocks of 256 x 256, 14 parts each) keeps the bound on
    the length of a sum in tensor-core accumulators (24 K blocks).  A A^T X
    alone (one iteration, (a, b, c) = (0, 1, 0)) on some columns against fp64:
    the products of K = 20480 of APPLY, which are not cut, leave 2.5e-5; with
    whole Gram tiles (320 K blocks) it was 7.6e-5."""
    import torch
    from paper_2605_19811_gb300 import lionmuon as L
    n = 20480
    gen = torch.Generator(device="cuda")
    gen.manual_seed(2)
    x = torch.randn((n, n), generator=gen, device="cuda")
    out = torch.empty_like(x)
    L.msign_ns(x, out, 1, 0.0, 1.0, 0.0, precision=L.LM_NS_F32_TC)
    rows = [x[i:i + 2048] for i in range(0, n, 2048)]
    v = sum(r.double().t() @ r[:, :64].double() for r in rows)
    norm = sum(float(r.double().square().sum()) for r in rows) ** 0.5
    want = torch.cat([r.double() @ v for r in rows]) / (norm + 1e-7) ** 3
    assert float((out[:, :64].double() - want).norm() / want.norm()) <= 4e-5


@pytest.mark.parametrize("precision", [0, 2])
def test_fp32_chain_from_a_graph_and_sharded(precision):
    """The fp32 modes replayed from a CUDA graph equal eager steps; two sharded
    states, each with the tiles of its own matrices, give the single state's
    parameters within the modes' error (Gram tiles are cut otherwise)."""
    import torch
    from paper_2605_19811_gb300 import lionmuon as L
    from paper_2605_19811_gb300 import shard
    shapes = [(512, 640), (1400, 512), (640, 512), (512, 1400)]
    cfg = dict(period=1, eta_muon=0.02, ns_precision=precision)
    grads = [host_tensor(x, "f32").cuda() for x in synth.draw_grads(shapes, "student_t", seed=0, step=0)]

    def fresh(**kw):
        p = [host_tensor(w, "f32").cuda() for w in synth.init_weights(shapes, seed=1)]
        return p, L.LionMuon(p, **cfg, **kw)
    eager, opt = fresh()
    replayed, graphed = fresh()
    graph = graphed.capture_steps(grads)[0]
    for t in range(2):
        opt.step(grads, t)
        graph.replay()
    own = shard.owners(shapes, 2)
    ranks = [fresh(shard_rank=r, shard_world=2) for r in range(2)]
    for t in range(2):
        for p, o in ranks:
            o.step(grads, t)
        for i, r in enumerate(own):
            ranks[1 - r][0][i].copy_(ranks[r][0][i])
    torch.cuda.synchronize()
    for o in (opt, graphed, ranks[0][1], ranks[1][1]):
        assert o.status() == 0 and o.ns_path() == L.LM_NS_F32_TC
    assert sorted(set(own)) == [0, 1]
    for i in range(len(shapes)):
        np.testing.assert_array_equal(bits(replayed[i]), bits(eager[i]))
        for p, _ in ranks:   # the update is a few percent of W, each within 2e-5
            assert rel_fro(stored_values(p[i]), stored_values(eager[i])) <= 4e-6


# ------------------------- beside other work -------------------------------
def test_step_beside_another_streams_kernel():
    """The chain needs its SMs at the same time; a kernel of another stream
    that holds one delays it and changes nothing."""
    import torch
    from paper_2605_19811_gb300 import lionmuon as L
    shapes = [(768, 768), (768, 3072), (3072, 768)]
    grads = [host_tensor(x, "bf16").cuda() for x in synth.draw_grads(shapes, "student_t", seed=0, step=0)]
    got = []
    for busy in (False, True):
        params = [host_tensor(w, "bf16").cuda() for w in synth.init_weights(shapes, seed=1)]
        opt = L.LionMuon(params, period=1)
        other = torch.cuda.Stream()
        torch.cuda.synchronize()
        for t in range(3):
            if busy:
                with torch.cuda.stream(other):
                    torch.cuda._sleep(2_000_000)   # about a millisecond on one SM
            opt.step(grads, t)
        torch.cuda.synchronize()
        assert opt.status() == 0
        got.append([bits(p) for p in params])
        opt.close()
    for x, y in zip(*got):
        np.testing.assert_array_equal(x, y)


@pytest.fixture
def green_stream():
    """A stream on 32 of the device's SMs (a green context)."""
    import ctypes
    import torch
    torch.zeros(1, device="cuda")
    cu = ctypes.CDLL("libcuda.so.1")
    res, part, rest = (ctypes.create_string_buffer(256) for _ in range(3))   # CUdevResource is 144 bytes
    n, desc, ctx, stream = ctypes.c_uint(1), ctypes.c_void_p(), ctypes.c_void_p(), ctypes.c_void_p()
    sm = 1                                                                   # CU_DEV_RESOURCE_TYPE_SM
    if (cu.cuDeviceGetDevResource(0, res, sm) or cu.cuDevSmResourceSplitByCount(part, ctypes.byref(n), res, rest, 0, 32)
            or cu.cuDevResourceGenerateDesc(ctypes.byref(desc), part, 1)
            or cu.cuGreenCtxCreate(ctypes.byref(ctx), desc, 0, 1) or cu.cuGreenCtxStreamCreate(ctypes.byref(stream), ctx, 1, 0)):
        pytest.skip("no green contexts")
    yield torch.cuda.ExternalStream(stream.value)
    assert cu.cuStreamSynchronize(stream) == 0
    cu.cuStreamDestroy_v2(stream)
    cu.cuGreenCtxDestroy(ctx)


@pytest.mark.parametrize("precision,dtype,shapes,cfg", [
    (1, "bf16", [(768, 768), (20000, 768), (768, 2304), (768,)], {}),    # Gram tiles split along K
    (1, "bf16", [(512, 1024), (1024, 512)] * 3, dict(schedule=1, srank_alpha=0.02)),
    (1, "bf16", [(512, 640), (640, 512)], dict(ns_coeffs=((4.1, -3.1, 0.6), (1.5, -0.5, 0.0)))),   # a cubic last
    (2, "f32", [(768, 768), (20000, 768)], {}),
    (0, "f32", [(1024, 1024), (1100, 9000)], {})])
def test_part_of_the_device(precision, dtype, shapes, cfg, green_stream):
    """Steps on a stream that has fewer SMs than the state was planned for run
    there (a launch per phase, none of which waits for another pair), with the
    same results; the static-area msign too."""
    import torch
    from paper_2605_19811_gb300 import lionmuon as L
    cfg = dict(period=1, **cfg) if "schedule" not in cfg else cfg
    grads = [[host_tensor(x, dtype).cuda() for x in synth.draw_grads(shapes, "student_t", seed=0, step=t)] for t in range(2)]
    got = []
    for stream in (None, green_stream):
        params = [host_tensor(w, dtype).cuda() for w in synth.init_weights(shapes, seed=1)]
        x = host_tensor(synth.draw_matrix((768, 2048), seed=3), "bf16").cuda()
        out = torch.empty((768, 2048), device="cuda")
        torch.cuda.synchronize()
        opt = L.LionMuon(params, stream=stream, ns_precision=precision, **cfg)
        for t in range(2):
            opt.step(grads[t], t, stream=stream)
        L.msign_ns_noalloc(x, out, stream=stream)
        assert L.msign_ns_noalloc_status(stream=stream) == (0, 0)
        assert opt.status() == 0
        torch.cuda.synchronize()
        got.append([bits(p) for p in params] + [bits(opt.momentum(i)) for i in range(len(params))] + [bits(out)])
        opt.close()
    for a, b in zip(*got):
        np.testing.assert_array_equal(a, b)
