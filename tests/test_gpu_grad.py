"""GPU parity of the two gradient maps of the projection (dX, dW) against the fp64 oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2609_32814_b200 import binding, synth
from tests import helpers as H

pytestmark = pytest.mark.gpu


def _problem(q, M, s_w, r_w, types=None, integer=True, seed=1):
    if types is None:
        types = synth.uniform_types(5000 + seed, M, q)
    wl = synth.make_workload("grad", config=8, variant=500 + seed, dtype="bf16", q=q, M=M, D=s_w * q, F=r_w * q, types=types,
                             integer=integer, with_down=False)
    G = synth.small_ints(synth.seed_for(8, 900 + seed), (M, r_w * q)) if integer else \
        synth.bf16_round(synth.normal(synth.seed_for(8, 900 + seed), (M, r_w * q), 1.0))
    return wl, G


@pytest.mark.parametrize("q,M,s_w,r_w,schedule", [
    (2, 300, 128, 128, "explicit"),     # one tile per block, ragged buckets
    (2, 1000, 384, 256, "explicit"),    # several tiles, both endpoint products
    (3, 515, 128, 256, "explicit"),     # non-power-of-two q
    (4, 777, 128, 512, "explicit"),     # config-3 group shapes
    (1, 200, 256, 256, "explicit"),     # q = 1: the gradients of an ordinary GEMM
    (2, 1024, 256, 128, "cyclic"),      # cyclic schedule, whole 64-row blocks per type: X and G read in place
    (4, 4 * 192, 128, 384, "cyclic"),   # in place, three reduction blocks per type, four segments on the diagonal
    (3, 3 * 64, 384, 128, "cyclic"),    # in place, one block per type, several feature tiles
    (2, 1000, 128, 256, "cyclic"),      # 500 rows per type: not whole blocks, padded copies
])
def test_grad_maps_integer_bit_exact(q, M, s_w, r_w, schedule):
    types = synth.cyclic_types(M, q) if schedule == "cyclic" else None
    wl, G = _problem(q, M, s_w, r_w, types=types, seed=q * 7 + M % 5)
    g = binding.ProjGrad(wl.d_widths, wl.f_widths, schedule=schedule)
    t = None if schedule == "cyclic" else H.dev_types(wl.types)
    Xd, Wd, Gd = H.to_dev(wl.X, "bf16"), H.to_dev(wl.W_up, "bf16"), H.to_dev(G, "bf16")
    dX = g.grad_input(Gd, t, Wd, out_dtype=torch.float32)
    dW = g.grad_weight(Xd, Gd, t)
    assert g.last_status() == 0
    ref_dx = oracle.proj_vjp_x(G, wl.types, wl.W_up, wl.d_widths, wl.f_widths)
    ref_dw = oracle.proj_vjp_w(wl.X, G, wl.types, wl.d_widths, wl.f_widths)
    bad = np.argwhere(H.to_np(dX) != ref_dx)
    assert bad.size == 0, f"dX: {len(bad)} mismatches, first {bad[:5].tolist()}"
    bad = np.argwhere(H.to_np(dW) != ref_dw)
    assert bad.size == 0, f"dW: {len(bad)} mismatches, first {bad[:5].tolist()}"
    # repeatable bit for bit (one owner per output element, no atomics)
    assert torch.equal(dW, g.grad_weight(Xd, Gd, t)) and torch.equal(dX, g.grad_input(Gd, t, Wd, out_dtype=torch.float32))


def test_grad_tables_missing_type_and_bad_type():
    q, M, s_w, r_w = 4, 600, 128, 128
    wl, G = _problem(q, M, s_w, r_w, seed=9)
    Xd, Wd, Gd = H.to_dev(wl.X, "bf16"), H.to_dev(wl.W_up, "bf16"), H.to_dev(G, "bf16")
    for table in ("dense", "q2pow"):
        keep = oracle.support(q, table)
        g = binding.ProjGrad(wl.d_widths, wl.f_widths, table=table)
        assert np.array_equal(H.to_np(g.grad_input(Gd, H.dev_types(wl.types), Wd, out_dtype=torch.float32)),
                              oracle.proj_vjp_x(G, wl.types, wl.W_up, wl.d_widths, wl.f_widths, keep=keep)), table
        assert np.array_equal(H.to_np(g.grad_weight(Xd, Gd, H.dev_types(wl.types))),
                              oracle.proj_vjp_w(wl.X, G, wl.types, wl.d_widths, wl.f_widths, keep=keep)), table
    # a type with no rows: its private weight blocks get a zero gradient
    types = np.where(wl.types == 3, 1, wl.types).astype(np.int32)
    g = binding.ProjGrad(wl.d_widths, wl.f_widths)
    dW = H.to_np(g.grad_weight(Xd, Gd, H.dev_types(types)))
    assert np.array_equal(dW, oracle.proj_vjp_w(wl.X, G, types, wl.d_widths, wl.f_widths))
    assert not dW[3 * s_w:, :3 * r_w].any()
    # an out-of-range type: status raised, the row contributes to no block and gets a zero input gradient
    types[5] = 11
    dW = H.to_np(g.grad_weight(Xd, Gd, H.dev_types(types)))
    assert g.last_status() == 5
    good = np.ones(M, bool)
    good[5] = False
    assert np.array_equal(dW, oracle.proj_vjp_w(wl.X[good], G[good], types[good], wl.d_widths, wl.f_widths))
    dX = H.to_np(g.grad_input(Gd, H.dev_types(types), Wd, out_dtype=torch.float32))
    assert g.last_status() == 5 and not dX[5].any()
    assert np.array_equal(dX[good], oracle.proj_vjp_x(G[good], types[good], wl.W_up, wl.d_widths, wl.f_widths))


def test_grad_config2_up_projection_normal_data():
    """The up projection of configuration 2 (768 -> 3072, M = 8192, type = position mod 2), real-valued
    data: both gradients within the bf16 tolerance of the fp64 oracle (dW on a sample of its rows)."""
    wl = synth.config2()
    G = synth.bf16_round(synth.normal(synth.seed_for(2, 77), (wl.M, wl.F), 1.0))
    g = binding.ProjGrad(wl.d_widths, wl.f_widths, schedule="cyclic")
    Xd, Wd, Gd = H.to_dev(wl.X, "bf16"), H.to_dev(wl.W_up, "bf16"), H.to_dev(G, "bf16")
    dX = g.grad_input(Gd, None, Wd, out_dtype=torch.float32)
    dW = g.grad_weight(Xd, Gd, None)
    rows = np.arange(0, wl.M, 16)
    ref_dx = oracle.proj_vjp_x(G[rows], wl.types[rows], wl.W_up, wl.d_widths, wl.f_widths)
    got = H.to_np(dX[torch.from_numpy(rows).cuda()])
    assert H.rel_fro(got, ref_dx) <= H.BF16_REL_FRO and H.max_abs(got, ref_dx) <= H.BF16_MAX_ABS
    ref_dw = oracle.proj_vjp_w(wl.X, G, wl.types, wl.d_widths, wl.f_widths)
    got = H.to_np(dW)
    assert H.rel_fro(got, ref_dw) <= 1e-4        # exact bf16 products, fp32 accumulation over 4096-8192 rows
    assert np.abs(got - ref_dw).max() <= 2e-2 + 1e-4 * np.abs(ref_dw).max()


def test_grad_refusals():
    with pytest.raises(binding.AlgError) as e:
        binding.ProjGrad([64, 64], [72, 72])      # output groups the tensor-core tiles do not divide
    assert e.value.code == 2


@pytest.mark.parametrize("q,M,s_w,r_w,schedule", [
    (2, 1024, 384, 1536, "cyclic"),      # dW in place, 72 tiles of 256 columns
    (2, 1000, 384, 1536, "explicit"),    # dW through the padded copies, dX too
    (2, 300, 256, 256, "explicit"),      # four and eight CTAs per tile
    (4, 512, 128, 256, "cyclic"),
])
def test_grad_maps_on_split_reductions(q, M, s_w, r_w, schedule):
    types = synth.cyclic_types(M, q) if schedule == "cyclic" else synth.uniform_types(M, M, q)
    X, G = synth.small_ints(1, (M, q * s_w), -1, 1), synth.small_ints(2, (M, q * r_w), -1, 1)
    W = synth.small_ints(3, (q * s_w, q * r_w), -1, 1)
    grad = binding.ProjGrad([s_w] * q, [r_w] * q, schedule=schedule)
    tt = None if schedule == "cyclic" else H.dev_types(types)
    dX = grad.grad_input(H.to_dev(G, "bf16"), tt, H.to_dev(W, "bf16"), out_dtype=torch.float32)
    dW = grad.grad_weight(H.to_dev(X, "bf16"), H.to_dev(G, "bf16"), tt)
    assert grad.last_status() == 0
    widths = [s_w] * q, [r_w] * q
    assert np.array_equal(H.to_np(dX), oracle.proj_vjp_x(G, types, W, *widths))
    assert np.array_equal(H.to_np(dW), oracle.proj_vjp_w(X, G, types, *widths))


@pytest.mark.parametrize("q,M,s,r", [
    (2, 900, [200, 56], [128, 256]),     # feature groups on 16 bytes but off the tile: X through rows of 512 bytes
    (3, 515, [20, 44, 64], [128] * 3),   # feature groups off 16 bytes: X transposed
    (2, 70, [128, 128], [1280, 1280]),   # G rows of several pieces, few rows
])
@pytest.mark.parametrize("schedule", ["explicit", "cyclic"])
def test_weight_gradient_row_copies(q, M, s, r, schedule):
    M = M // q * q
    types = synth.cyclic_types(M, q) if schedule == "cyclic" else synth.uniform_types(M, M, q)
    X, G = synth.small_ints(1, (M, sum(s)), -1, 1), synth.small_ints(2, (M, sum(r)), -1, 1)
    grad = binding.ProjGrad(s, r, schedule=schedule)
    dW = grad.grad_weight(H.to_dev(X, "bf16"), H.to_dev(G, "bf16"), None if schedule == "cyclic" else H.dev_types(types))
    assert grad.last_status() == 0
    assert np.array_equal(H.to_np(dW), oracle.proj_vjp_w(X, G, types, s, r))


@pytest.mark.parametrize("q,M,s,r,schedule,bad", [
    (3, 130, [64, 136, 8], [2560, 256, 2048], "explicit", False),   # parts of a G row in several pieces, one of them around the gap
    (3, 130, [64, 136, 8], [2560, 256, 2048], "explicit", True),
    (2, 65, [128, 384], [1536, 1536], "explicit", False),           # one row past whole blocks, clusters of CTAs per tile
    (2, 65, [128, 384], [1536, 1536], "explicit", True),
    (2, 1, [128, 128], [256, 256], "explicit", False),              # a single row
    (2, 1, [128, 128], [256, 256], "explicit", True),
    (2, 2050, [1024, 1024], [4096, 4096], "explicit", False),       # more tiles than CTAs: the persistent kernel
    (2, 2050, [1024, 1024], [4096, 4096], "explicit", True),
    (4, 3 * 100, [64, 72, 80, 200], [128] * 4, "cyclic", False),    # 75 rows per type: not read in place
    (32, 700, [128] * 32, [128] * 32, "explicit", False),           # slots that whole rows may widen: X and G rows of one piece
    (32, 700, [128] * 32, [128] * 32, "explicit", True),
    (16, 300, [8] * 16, [640] * 16, "explicit", True),              # whole rows in more pieces than their parts
])
def test_weight_gradient_blocks_that_take_every_row(q, M, s, r, schedule, bad):
    """dW_kk is reduced over X and G as they lie, the other blocks over the parts of the rows that were copied; a batch with
    a type out of range takes everything from whole copies."""
    types = synth.cyclic_types(M, q) if schedule == "cyclic" else synth.uniform_types(M, M, q)
    good = np.ones(M, bool)
    if bad:
        types = types.copy()
        types[M // 2], good[M // 2] = q, False
    X, G = synth.small_ints(1, (M, sum(s)), -1, 1), synth.small_ints(2, (M, sum(r)), -1, 1)
    grad = binding.ProjGrad(s, r, schedule=schedule)
    ws = torch.full((grad.workspace_bytes(M),), 0xFF, dtype=torch.uint8, device="cuda")   # what is not copied is NaN
    dW = grad.grad_weight(H.to_dev(X, "bf16"), H.to_dev(G, "bf16"), None if schedule == "cyclic" else H.dev_types(types), workspace=ws)
    assert grad.last_status() == (5 if bad else 0)
    assert np.array_equal(H.to_np(dW), oracle.proj_vjp_w(X[good], G[good], types[good], s, r))


@pytest.mark.parametrize("M,s,r", [
    (60, [20, 44, 64], [128] * 3),       # one CTA per tile
    (2000, [20, 44, 64], [128] * 3),     # clusters of CTAs per tile
    (70, [1028, 1020], [4096] * 2),      # more tiles than CTAs: an accumulator holds the sums of the tile before
    (70, [1024, 1024], [4096] * 2),      # the same with feature groups on 16 bytes: X as it is
])
@pytest.mark.parametrize("rows_of", [[0], [1], []])
def test_weight_gradient_blocks_without_rows(M, s, r, rows_of):
    """Blocks that no row of the batch belongs to are zero, whatever tensor memory held before: all rows of one type, and
    no row of any."""
    q = len(s)
    wide = binding.ProjGrad([1024, 1024], [4096] * 2)   # leaves sums in the tensor memory of every SM
    ones = torch.ones((64, 8192), dtype=torch.bfloat16, device="cuda")
    wide.grad_weight(ones[:, :2048].contiguous(), ones, torch.zeros(64, dtype=torch.int32, device="cuda"))
    types = np.full(M, rows_of[0] if rows_of else q, np.int32)
    X, G = synth.small_ints(1, (M, sum(s)), -1, 1), synth.small_ints(2, (M, sum(r)), -1, 1)
    grad = binding.ProjGrad(s, r)
    dW = H.to_np(grad.grad_weight(H.to_dev(X, "bf16"), H.to_dev(G, "bf16"), H.dev_types(types)))
    assert grad.last_status() == (0 if rows_of else 5)
    ref = oracle.proj_vjp_w(X, G, types, s, r) if rows_of else np.zeros(dW.shape)
    assert np.array_equal(dW, ref)


@pytest.mark.parametrize("q,M,s,r,schedule", [
    (2, 300, [128, 128], [256, 256], "explicit"),        # clusters of CTAs per tile
    (2, 70, [1024, 1024], [4096, 4096], "explicit"),     # one CTA per tile
    (3, 515, [20, 44, 64], [128] * 3, "explicit"),       # X transposed
    (2, 512, [128, 256], [128, 384], "cyclic"),          # X and G in place
])
def test_weight_gradient_of_strided_operands(q, M, s, r, schedule):
    """X, G and a bf16 dW inside wider allocations; of explicit types also with one out of range."""
    all_types = synth.cyclic_types(M, q) if schedule == "cyclic" else synth.uniform_types(M, M, q)
    K, N = sum(s), sum(r)
    X, G = synth.small_ints(1, (M, K), -1, 1), synth.small_ints(2, (M, N), -1, 1)
    Xp = torch.full((M, K + 24), float("nan"), dtype=torch.bfloat16, device="cuda")
    Gp = torch.full((M, N + 8), float("nan"), dtype=torch.bfloat16, device="cuda")
    Xp[:, :K], Gp[:, :N] = H.to_dev(X, "bf16"), H.to_dev(G, "bf16")
    grad = binding.ProjGrad(s, r, schedule=schedule)
    for bad in [False, True] if schedule == "explicit" else [False]:
        types, good = all_types.copy(), np.ones(M, bool)
        if bad:
            types[M // 3], good[M // 3] = q, False
        out = torch.full((K, N + 16), 7.0, dtype=torch.bfloat16, device="cuda")
        grad.grad_weight(Xp[:, :K], Gp[:, :N], None if schedule == "cyclic" else H.dev_types(types), out=out[:, :N])
        assert grad.last_status() == (5 if bad else 0)
        ref = H.bf16_rne(oracle.proj_vjp_w(X[good], G[good], types[good], s, r))
        assert np.array_equal(H.to_np(out[:, :N].contiguous()), ref)
        assert torch.all(out[:, N:] == 7.0)


@pytest.mark.parametrize("schedule", ["explicit", "cyclic"])
@pytest.mark.parametrize("over", ["X", "G"])
def test_weight_gradient_over_an_operand(schedule, over):
    """dW in the memory of X or G: more tiles than CTAs, so that tiles reduce after others have been stored."""
    q, M, s, r = 2, 512, [512, 512], [5120, 5120]
    K, N = sum(s), sum(r)
    types = synth.cyclic_types(M, q) if schedule == "cyclic" else synth.uniform_types(M, M, q)
    X, G = synth.small_ints(1, (M, K), -1, 1), synth.small_ints(2, (M, N), -1, 1)
    room = torch.empty(max(M, K) * N, dtype=torch.bfloat16, device="cuda")
    Xd, Gd = H.to_dev(X, "bf16"), H.to_dev(G, "bf16")
    if over == "X":
        Xd = room[:M * K].view(M, K).copy_(Xd)
    else:
        Gd = room[:M * N].view(M, N).copy_(Gd)
    grad = binding.ProjGrad(s, r, schedule=schedule)
    dW = grad.grad_weight(Xd, Gd, None if schedule == "cyclic" else H.dev_types(types), out=room[:K * N].view(K, N))
    assert grad.last_status() == 0
    assert np.array_equal(H.to_np(dW), H.bf16_rne(oracle.proj_vjp_w(X, G, types, s, r)))
