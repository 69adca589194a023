"""Sizes at which the kernels change form: one step against the float64 oracle, or a matrix against its own bits in
another form of the same call."""
import numpy as np
import pytest
import torch

from oracle import orthdion_oracle as orc
from paper_2605_16341_b200 import binding as od
from paper_2605_16341_b200 import workloads as wl
from parity_util import TOL_STEP, GpuMatrix, f64, poisoned_workspace, rel
from test_gpu_parity import make_problem, one_step_compare

pytestmark = pytest.mark.gpu
F32, BF16 = torch.float32, torch.bfloat16
MODES = [od.MODE_ORTH, od.MODE_COLNORM]


# the one-kernel QR on the fp32 engine: each width of its ranks and the first beyond, ranks that are no multiple of four, one
# row past a part, last CTAs of the cluster without rows, more rows than the tensor engine gives it
@pytest.mark.parametrize("shape", [(40, 33, 3), (257, 300, 16), (129, 700, 17), (1025, 70, 33), (100, 1301, 63), (900, 1100, 64), (300, 200, 65)])
@pytest.mark.parametrize("mode", MODES)
def test_one_kernel_qr_of_the_fp32_engine(shape, mode):
    m, n, r = shape
    spec, X, M, G, Q = make_problem(m, n, r, F32, BF16, seed=m + n + r)
    one_step_compare(spec, X, M, G, Q, mode=mode, engine=od.ENGINE_SIMT)


# Q1 of the first pass 1e-4 to 1.4e-3 away from orthonormal: two columns of Y all but parallel, 96 draws.  A first-order inverse in the second
# pass leaves out up to 0.75 times the square of that, 1.5e-6; rounding alone stays below eight halves of a spacing at 1 (2^-24)
@pytest.mark.parametrize("case", [(200, 100, 9, 0.012), (200, 100, 9, 0.02), (150, 304, 30, 0.012)])
def test_fp32_engine_is_orthonormal_to_rounding(case):
    m, n, r, eps = case
    count = 96
    gen = torch.Generator().manual_seed(m + n + r)
    h = od.orthdion_create(m, n, r, 0.95, 0.01, 0.0, od.MODE_ORTH)
    od.orthdion_set_dtypes(h, F32, F32)
    od.orthdion_set_engine(h, od.ENGINE_SIMT)
    G, Q = [], []
    for _ in range(count):
        Y = torch.randn(m, r, generator=gen)
        Y[:, 1] = Y[:, 0] + eps * Y[:, 1]
        Q.append(wl.random_orthonormal(n, r, gen).cuda())
        G.append(Y.cuda() @ Q[-1].T)
    X, M = ([torch.zeros(m, n, device="cuda") for _ in range(count)] for _ in range(2))
    ws = poisoned_workspace(od.orthdion_workspace_bytes_grouped([h] * count))
    od.orthdion_step_grouped(od.PointerTable([h] * count, X, M, G, Q), ws)
    torch.cuda.synchronize()
    worst = 0.0
    for i in range(count):
        for A in (od.orthdion_get_factors([h] * count, i, ws, (m, n, r))[0].double(), Q[i].double()):
            worst = max(worst, (A.T @ A - torch.eye(r, device="cuda", dtype=torch.float64)).abs().max().item())
    assert worst <= 8 * 2.0 ** -24
    od.orthdion_destroy(h)


# its 512-thread form (parts of 256 rows and more): the last size below, the first, a ragged one
@pytest.mark.parametrize("shape", [(3584, 136, 32), (3585, 136, 32), (7700, 264, 16)])
@pytest.mark.parametrize("mode", MODES)
def test_one_kernel_qr_of_long_parts(shape, mode):
    m, n, r = shape
    spec, X, M, G, Q = make_problem(m, n, r, F32, F32, seed=m + n + r)
    one_step_compare(spec, X, M, G, Q, mode=mode, engine=od.ENGINE_TENSOR)


# rows that only its 256-thread form has room for, up to the last ones: six launches still
@pytest.mark.parametrize("case", [(24320, 136, 32, od.ENGINE_TENSOR), (26112, 72, 32, od.ENGINE_TENSOR), (39700, 40, 16, od.ENGINE_TENSOR),
                                  (11263, 71, 41, od.ENGINE_SIMT), (26111, 60, 18, od.ENGINE_SIMT)])
def test_one_kernel_qr_up_to_its_last_rows(case):
    m, n, r, engine = case
    spec, X, M, G, Q = make_problem(m, n, r, BF16, F32, seed=m)
    before = od.orthdion_launch_count()
    one_step_compare(spec, X, M, G, Q, mode=od.MODE_ORTH, engine=engine)
    assert od.orthdion_launch_count() == before + 6


# a call of six kernels on either side of the size up to which its launches overlap
@pytest.mark.parametrize("shape", [(4096, 2048, 32), (4104, 2048, 32)])
def test_steps_back_to_back_at_the_largest_overlapping_size(shape):
    m, n, r = shape
    spec, X, M, G, Q = make_problem(m, n, r, BF16, BF16, seed=m)
    one_step_compare(spec, X, M, G, Q, mode=od.MODE_ORTH, engine=od.ENGINE_TENSOR)
    pair = [GpuMatrix(spec, X, M, Q, mu=0.95, eta=0.01, engine=od.ENGINE_TENSOR) for _ in range(2)]
    grad = G.cuda()
    for gm in pair:
        for _ in range(4):
            od.orthdion_step(gm.h, gm.X, gm.M, grad, gm.Q, gm.ws)
            if gm is pair[0]:
                torch.cuda.synchronize()
        torch.cuda.synchronize()
    assert all(torch.equal(getattr(pair[0], k), getattr(pair[1], k)) for k in "XMQ")
    for gm in pair:
        gm.close()


# the fused pass where the R and Q pieces have slots of their own (split terms of both, or fp32 G or X) and where they share
# one: a single 16-deep slice, a ragged last depth block, a last tile of 8 columns
@pytest.mark.parametrize("shape", [(300, 264, 16), (260, 392, 80), (600, 136, 128)])
@pytest.mark.parametrize("passes", [(1, 1), (3, 1), (1, 3), (3, 3)])
@pytest.mark.parametrize("dt", [(F32, F32), (F32, BF16), (BF16, F32), (BF16, BF16)])
def test_fused_pass_slots(shape, passes, dt):
    m, n, r = shape
    spec, X, M, G, Q = make_problem(m, n, r, *dt, seed=m + n + r)
    gm = GpuMatrix(spec, X, M, Q, mu=0.95, eta=0.01, engine=od.ENGINE_TENSOR, passes={2: passes[0], 3: passes[1]})
    gm.step(G)
    assert gm.status() == 0
    P, R = (f64(t) for t in gm.factors())
    Qn = f64(gm.Q)
    # what one product loses: two roundings of 2^-9 (bf16) or 2^-12 (fp16, both passes single) per term, or what two bf16
    # terms leave out; then fp32 arithmetic (1e-4 of the quotient by b = 0.05)
    lost = [2.0 ** -15 if p == 3 else 2.0 ** -11 if passes == (1, 1) else 2.0 ** -8 for p in passes]
    assert rel((f64(M) + f64(G) - f64(gm.M)) / 0.05, P @ R.T) <= lost[0] + 1e-4
    want = f64(X) - 0.01 * (P @ Qn.T)
    if dt[0] == F32:
        assert rel(f64(gm.X) - f64(X), want - f64(X)) <= lost[1] + 1e-4
    else:                       # the stored weight, half a spacing and the product's loss away
        far = 0.01 * 2 * lost[1] * np.linalg.norm(P, axis=1)[:, None] * np.linalg.norm(Qn, axis=1)[None, :]
        assert (np.abs(f64(gm.X) - want) <= 2.0 ** -8 * np.abs(want) + far).all()
    gm.close()


def _grouped(specs, probs, hs, lanes):
    """X, M, Q after one grouped step on `lanes` internal streams, and the status words."""
    X, M, G, Q = ([p[j].cuda() for p in probs] for j in (1, 2, 3, 4))
    ws = poisoned_workspace(od.orthdion_workspace_bytes_grouped(hs))
    od.orthdion_set_concurrency(lanes)
    try:
        od.orthdion_step_grouped(od.PointerTable(hs, X, M, G, Q), ws)
        torch.cuda.synchronize()
    finally:
        od.orthdion_set_concurrency(4)
    return X, M, Q, od.orthdion_last_status(hs, ws)


@pytest.mark.parametrize("r", [128, 272])
def test_merged_factorisations_of_one_stream_leave_the_same_bits(r):
    # 155 matrices of two shapes: on one stream their factorisations are one launch (two CTAs per multiprocessor), on
    # several one per shape
    shapes = [(300, 320, r)] * 80 + [(320, 280, r)] * 75
    probs = [make_problem(*s, BF16, BF16, seed=50 + i) for i, s in enumerate(shapes)]
    plans = {s: od.orthdion_create(*s, 0.95, 0.01, 0.0, od.MODE_ORTH) for s in set(shapes)}
    hs = [plans[s] for s in shapes]
    one, many = (_grouped(shapes, probs, hs, lanes) for lanes in (1, 4))
    assert one[3] == many[3] == [0] * len(hs)
    for a, b in zip(one[:3], many[:3]):
        assert all(torch.equal(x, y) for x, y in zip(a, b))
    for i in (0, len(hs) - 1):                      # one of either shape
        _, X, M, G, Q = probs[i]
        ref = orc.step(f64(X), f64(M), f64(G), f64(Q), eta=0.01, mu=0.95, wd=0.0, mode=orc.ORTH)
        assert rel(f64(one[2][i]), ref["Q"]) <= TOL_STEP and rel(f64(one[1][i]), ref["M"]) <= TOL_STEP
    for h in plans.values():
        od.orthdion_destroy(h)


# more matrices of one plan than the smaller launch table holds: no more launches, and every matrix the bits that it gets alone
@pytest.mark.parametrize("case", [(96, 104, 32, od.MODE_ORTH, od.ENGINE_TENSOR, 0), (200, 160, 80, od.MODE_COLNORM, od.ENGINE_TENSOR, 3),
                                  (160, 144, 96, od.MODE_ORTH, od.ENGINE_TENSOR, 1), (90, 77, 24, od.MODE_ORTH, od.ENGINE_SIMT, 1),
                                  (110, 120, 70, od.MODE_ORTH, od.ENGINE_SIMT, 0), (110, 121, 70, od.MODE_COLNORM, od.ENGINE_SIMT, 0)])
def test_more_matrices_than_the_smaller_launch_table(case):
    m, n, r, mode, engine, diag = case
    probs = [make_problem(m, n, r, F32, BF16, seed=i) for i in range(132)]
    h = od.orthdion_create(m, n, r, 0.95, 0.01, 0.0, mode)
    od.orthdion_set_dtypes(h, F32, BF16)
    od.orthdion_set_engine(h, engine)
    od.orthdion_set_diagnostics(h, diag)
    launches = []
    for count, lanes in ((128, 1), (132, 1), (132, 4)):
        before = od.orthdion_launch_count()
        X, M, Q, flags = _grouped(None, probs[:count], [h] * count, lanes)
        launches.append(od.orthdion_launch_count() - before)
        assert flags == [0] * count
        for i in (0, 65, 66, 127, count - 1):
            spec, x, mm, g, q = probs[i]
            gm = GpuMatrix(spec, x, mm, q, mu=0.95, eta=0.01, mode=mode, engine=engine)
            gm.step(g)
            assert torch.equal(gm.X, X[i]) and torch.equal(gm.M, M[i]) and torch.equal(gm.Q, Q[i])
            gm.close()
    assert launches[1] == launches[0]
    od.orthdion_destroy(h)


@pytest.mark.parametrize("r", [96, 256, 272])
def test_third_pass_of_one_matrix_among_others(r):
    """Products of a third pass look at the status words of their launch first: the one matrix that asked for the pass gets
    it, and every matrix the bits that it gets alone."""
    m, n = 640, 520
    probs = [make_problem(m, n, r, F32, F32, seed=300 + i) for i in range(4)]
    gen = torch.Generator().manual_seed(5)
    U, V = wl.random_orthonormal(m, r, gen), wl.random_orthonormal(n, r, gen)
    spec = probs[2][0]
    ill = ((U * torch.logspace(0, -5, r)[None, :]) @ V.T).contiguous()
    probs[2] = (spec, torch.zeros(m, n), torch.zeros(m, n), ill, V)
    h = od.orthdion_create(m, n, r, 0.95, 0.01, 0.0, od.MODE_ORTH)
    od.orthdion_set_dtypes(h, F32, F32)
    X, M, Q, flags = _grouped(None, probs, [h] * 4, 4)
    assert flags[2] & od.STATUS_SHIFTED_LEFT and [flags[i] for i in (0, 1, 3)] == [0, 0, 0]
    for i in range(4):
        spec, x, mm, g, q = probs[i]
        gm = GpuMatrix(spec, x, mm, q, mu=0.95, eta=0.01, engine=od.ENGINE_TENSOR)
        gm.step(g)
        assert gm.status() == flags[i]
        assert torch.equal(gm.X, X[i]) and torch.equal(gm.M, M[i]) and torch.equal(gm.Q, Q[i])
        gm.close()
    od.orthdion_destroy(h)


# the eigenvalue iteration of the diagnostics: each size of its cluster, a last CTA with fewer rows, rows in memory (r = 656),
# a rank that is no multiple of four
@pytest.mark.parametrize("case", [(300, 320, 144, od.ENGINE_TENSOR), (400, 304, 272, od.ENGINE_TENSOR), (500, 480, 432, od.ENGINE_TENSOR),
                                  (700, 680, 656, od.ENGINE_TENSOR), (300, 281, 259, od.ENGINE_SIMT)])
def test_largest_singular_value_of_q(case):
    m, n, r, engine = case
    spec, X, M, G, Q = make_problem(m, n, r, F32, F32, seed=m + n + r)
    gm = GpuMatrix(spec, X, M, Q, mu=0.95, eta=0.01, mode=od.MODE_COLNORM, engine=engine)
    od.orthdion_set_diagnostics(gm.h, 1)
    gm.step(G)
    nu = od.orthdion_last_diagnostics([gm.h], gm.ws)[0]["nu"]
    want = float(torch.linalg.matrix_norm(gm.Q.double(), 2))
    assert abs(nu - want) <= 1e-3 * want            # the bound of every other test of nu (largest Ritz value after at most 96 steps)
    gm.close()


# a plan that fits the built-in scratch only without the partial Gram matrices: one CTA adds their chunks up, to the same bits
@pytest.mark.parametrize("shape", [(27904, 1024, 128), (30080, 520, 96)])
def test_gram_chunks_without_partial_matrices(shape):
    m, n, r = shape
    gen = torch.Generator(device="cuda").manual_seed(m)
    X, G = (torch.randn(m, n, generator=gen, device="cuda").bfloat16() for _ in range(2))
    M = torch.randn(m, n, generator=gen, device="cuda")
    Q = torch.linalg.qr(torch.randn(n, r, generator=gen, device="cuda"))[0].contiguous()
    h = od.orthdion_create(m, n, r, 0.95, 0.01, 0.0, od.MODE_ORTH)
    # (sixteen chunks of more than 64 depth blocks: with their partial matrices it would not fit)
    assert od.NOALLOC_SCRATCH_BYTES - 16 * r * r * 4 < od.orthdion_workspace_bytes(h) <= od.NOALLOC_SCRATCH_BYTES
    ws = poisoned_workspace(2 * od.NOALLOC_SCRATCH_BYTES)
    a, b = ([t.clone() for t in (X, M, Q)] for _ in range(2))
    od.orthdion_step(h, a[0], a[1], G, a[2], ws)
    od.orthdion_step_noalloc(h, b[0], b[1], G, b[2], None)
    torch.cuda.synchronize()
    assert od.orthdion_last_status([h], ws) == [0]
    assert all(torch.equal(x, y) for x, y in zip(a, b))
    od.orthdion_destroy(h)
