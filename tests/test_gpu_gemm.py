"""The two product engines against a plain PyTorch fp32 product of the same (rounded) inputs."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2609_21102_b200 import binding
    c = binding.Context(0)
    yield c
    c.close()


def _ref(A, B, ta, tb, alpha=1.0):
    a = A.float().transpose(1, 2) if ta else A.float()
    b = B.float().transpose(1, 2) if tb else B.float()
    return alpha * torch.matmul(a.double(), b.double()).float()


def _mk(b, r, c, dtype, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn((b, r, c), generator=g, device="cuda", dtype=torch.float32).to(dtype)


SHAPES = [(1, 128, 128, 64), (2, 200, 136, 96), (3, 256, 264, 200), (1, 72, 48, 40), (2, 384, 160, 320)]


@pytest.mark.parametrize("b,M,N,K", SHAPES)
@pytest.mark.parametrize("ta,tb", [(False, True), (False, False), (True, False), (True, True)])
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
def test_simt_engine(ctx, b, M, N, K, ta, tb, dtype):
    from paper_2609_21102_b200 import binding
    A = _mk(b, K if ta else M, M if ta else K, dtype, 1)
    B = _mk(b, N if tb else K, K if tb else N, dtype, 2)
    C = ctx.defl_debug_gemm(A, B, ta, tb, engine=binding.ENGINE_SIMT, out_dtype=torch.float32, alpha=0.5)
    ref = _ref(A, B, ta, tb, 0.5)
    assert torch.allclose(C, ref, rtol=1e-4, atol=1e-3)


@pytest.mark.parametrize("b,M,N,K", SHAPES)
@pytest.mark.parametrize("ta,tb", [(False, True), (False, False), (True, False), (True, True)])
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
def test_tensor_engine(ctx, b, M, N, K, ta, tb, dtype):
    from paper_2609_21102_b200 import binding
    A = _mk(b, K if ta else M, M if ta else K, dtype, 3)
    B = _mk(b, N if tb else K, K if tb else N, dtype, 4)
    if dtype == torch.float32 and (ta or not tb):
        # tf32 tiles are K-major only: the engine must refuse, not compute something else
        with pytest.raises(binding.DeflError) as e:
            ctx.defl_debug_gemm(A, B, ta, tb, engine=binding.ENGINE_TENSOR, out_dtype=torch.float32)
        assert e.value.code == -4
        return
    C = ctx.defl_debug_gemm(A, B, ta, tb, engine=binding.ENGINE_TENSOR, out_dtype=torch.float32)
    torch.cuda.synchronize()
    ref = _ref(A, B, ta, tb)
    if dtype == torch.bfloat16:      # exact products of bf16 values, fp32 accumulation
        assert torch.allclose(C, ref, rtol=1e-4, atol=2e-3)
    else:                            # tf32 operands: 10-bit mantissas
        err = (C - ref).norm() / ref.norm()
        assert err < 2e-3, float(err)


@pytest.mark.parametrize("n", [8, 16, 17, 32, 33, 65])
@pytest.mark.parametrize("k", [1, 15, 64, 65, 130])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16, torch.float16])
def test_simt_engine_tile_forms_and_operand_walks(ctx, n, k, dtype):
    """Every tile form (16, 32 and 64 columns wide) at its edges, with operands contiguous along K and along the rows,
    aligned for whole-quad loads and not. fp32 sums of k products: the bound is k rounding errors of 2^-24 each on the sum
    of the magnitudes (plus one for the store)."""
    from paper_2609_21102_b200 import binding
    for m in (31, 64, 132):
        for ta, tb in ((False, False), (True, True)):
            g = torch.Generator().manual_seed(1000 * n + 10 * k + m + ta)
            A = torch.randn((2, k, m) if ta else (2, m, k), generator=g).to(dtype).cuda()
            B = torch.randn((2, n, k) if tb else (2, k, n), generator=g).to(dtype).cuda()
            C = ctx.defl_debug_gemm(A, B, ta, tb, engine=binding.ENGINE_SIMT, out_dtype=torch.float32)
            Ad = A.double().transpose(1, 2) if ta else A.double()
            Bd = B.double().transpose(1, 2) if tb else B.double()
            bound = (k + 1) * 2.0 ** -24 * (Ad.abs() @ Bd.abs()) + 1e-30
            assert bool(((C.double() - Ad @ Bd).abs() <= bound).all()), (m, ta, tb)


def test_tensor_engine_bf16_output_and_large_tiles(ctx):
    from paper_2609_21102_b200 import binding
    A = _mk(2, 520, 1600, torch.bfloat16, 5)     # X X^T with a ragged 1600 = 12.5 tiles of 128
    C = ctx.defl_debug_gemm(A, A, False, True, engine=binding.ENGINE_TENSOR, out_dtype=torch.bfloat16)
    ref = _ref(A, A, False, True)
    err = (C.float() - ref).norm() / ref.norm()
    assert err < 4e-3, float(err)
    B = _mk(2, 1600, 1608, torch.bfloat16, 6)    # MN-major right operand, N = 1608 ragged
    A2 = _mk(2, 264, 1600, torch.bfloat16, 7)
    C2 = ctx.defl_debug_gemm(A2, B, False, False, engine=binding.ENGINE_TENSOR, out_dtype=torch.bfloat16)
    ref2 = _ref(A2, B, False, False)
    err2 = (C2.float() - ref2).norm() / ref2.norm()
    assert err2 < 4e-3, float(err2)


@pytest.mark.parametrize("b,M,N,K", [(2, 640, 200, 200), (1, 392, 136, 96), (2, 264, 72, 320), (1, 1600, 1600, 64)])
@pytest.mark.parametrize("ta,tb", [(True, True), (False, True), (True, False)])
@pytest.mark.parametrize("out_dtype", [torch.bfloat16, torch.float32])
def test_tensor_engine_transposed_output(ctx, b, M, N, K, ta, tb, out_dtype):
    """The product written transposed (the form the filter uses for X <- B X on a wide X): complete blocks take
    the coalesced path, ragged rows and columns the general one."""
    from paper_2609_21102_b200 import binding
    A = _mk(b, K if ta else M, M if ta else K, torch.bfloat16, 21)
    B = _mk(b, N if tb else K, K if tb else N, torch.bfloat16, 22)
    C = ctx.defl_debug_gemm(A, B, ta, tb, engine=binding.ENGINE_TENSOR, out_dtype=out_dtype, alpha=0.25, transpose_out=True)
    torch.cuda.synchronize()
    assert C.shape == (b, N, M)
    ref = _ref(A, B, ta, tb, 0.25).transpose(1, 2)
    if out_dtype == torch.float32:
        assert torch.allclose(C, ref, rtol=1e-4, atol=2e-3)
    else:
        assert torch.equal(C, ref.to(torch.bfloat16)) or float((C.float() - ref).norm() / ref.norm()) < 3e-3
    with pytest.raises(binding.DeflError) as e:      # the fp32 engine does not write transposed: refused, not ignored
        ctx.defl_debug_gemm(A, B, ta, tb, engine=binding.ENGINE_SIMT, out_dtype=out_dtype, transpose_out=True)
    assert e.value.code == -4


@pytest.mark.parametrize("engine_name", ["simt", "tensor"])
def test_symmetric_mirroring(ctx, engine_name):
    from paper_2609_21102_b200 import binding
    engine = binding.ENGINE_SIMT if engine_name == "simt" else binding.ENGINE_TENSOR
    A = _mk(2, 456, 320, torch.bfloat16, 8)
    C = ctx.defl_debug_gemm(A, A, False, True, engine=engine, out_dtype=torch.float32, exploit_symmetry=True)
    ref = _ref(A, A, False, True)
    assert torch.allclose(C, ref, rtol=1e-4, atol=2e-3)
    assert torch.equal(C, C.transpose(1, 2))


@pytest.mark.parametrize("knobs", [{"DEFL_TC_PAIR": "0"}, {"DEFL_TC_KSUB": "1"}, {"DEFL_TC_TILE_M": "128"},
                                   {"DEFL_TC_STAGES": "2"}, {"DEFL_TC_DYNAMIC": "1"},
                                   {"DEFL_TC_DYNAMIC": "1", "DEFL_TC_STAGES": "2"}])
@pytest.mark.parametrize("sym", [False, True])
def test_tensor_engine_other_tile_forms(monkeypatch, knobs, sym):
    """The tile forms the default rules do not pick for these shapes (single-CTA 256-row tile, one K block per
    stage, 128-row tiles, the shallowest pipeline) stay correct: a context reads the knobs when it is created."""
    from paper_2609_21102_b200 import binding
    for k, v in knobs.items():
        monkeypatch.setenv(k, v)
    ctx = binding.Context(0)
    A = _mk(2, 712, 1096, torch.bfloat16, 9)          # ragged in M (712 = 2 x 256 + 200), K = 17.1 blocks
    if sym:
        C = ctx.defl_debug_gemm(A, A, False, True, engine=binding.ENGINE_TENSOR, out_dtype=torch.float32,
                                exploit_symmetry=True)
        ref = _ref(A, A, False, True)
        assert torch.equal(C, C.transpose(1, 2))
    else:
        B = _mk(2, 1096, 328, torch.bfloat16, 10)     # MN-major right operand, ragged N
        C = ctx.defl_debug_gemm(A, B, False, False, engine=binding.ENGINE_TENSOR, out_dtype=torch.float32)
        ref = _ref(A, B, False, False)
    assert torch.allclose(C, ref, rtol=1e-4, atol=4e-3)


@pytest.mark.parametrize("K", [64, 200, 1096])
@pytest.mark.parametrize("sym", [False, True])
def test_tensor_engine_dynamic_tiles(monkeypatch, K, sym):
    """Tiles handed out through the counter (DEFL_TC_DYNAMIC), more tiles than CTA pairs so that every pair draws
    several; a one-step K, a short and a long one. Run twice: the counter must be back at zero after a launch."""
    from paper_2609_21102_b200 import binding
    monkeypatch.setenv("DEFL_TC_DYNAMIC", "1")
    ctx = binding.Context(0)
    A = _mk(14, 1000, K, torch.bfloat16, 31)
    B = A if sym else _mk(14, 1032, K, torch.bfloat16, 32)
    ref = _ref(A, B, False, True)
    for _ in range(2):
        C = ctx.defl_debug_gemm(A, B, False, True, engine=binding.ENGINE_TENSOR, out_dtype=torch.float32,
                                exploit_symmetry=sym)
        torch.cuda.synchronize()
        assert torch.allclose(C, ref, rtol=1e-4, atol=4e-3)


@pytest.mark.parametrize("ta,tb", [(False, True), (False, False), (True, False)])
@pytest.mark.parametrize("out_dtype", [torch.float16, torch.float32])
def test_tensor_engine_ieee_half(ctx, ta, tb, out_dtype):
    """IEEE half operands (the FP16 projection filter's type): exact products, fp32 accumulation."""
    from paper_2609_21102_b200 import binding
    b, M, N, K = 2, 328, 264, 200
    A = _mk(b, K if ta else M, M if ta else K, torch.float16, 21)
    B = _mk(b, N if tb else K, K if tb else N, torch.float16, 22)
    C = ctx.defl_debug_gemm(A, B, ta, tb, engine=binding.ENGINE_TENSOR, out_dtype=out_dtype)
    ref = _ref(A, B, ta, tb)
    if out_dtype == torch.float32:
        assert torch.allclose(C, ref, rtol=1e-4, atol=2e-3)
    else:
        assert torch.allclose(C.float(), ref, rtol=2.0 ** -10, atol=2e-3)      # one rounding to half on store
    As = _mk(b, 456, 320, torch.float16, 23)
    Cs = ctx.defl_debug_gemm(As, As, False, True, engine=binding.ENGINE_TENSOR, out_dtype=out_dtype, exploit_symmetry=True)
    assert torch.equal(Cs, Cs.transpose(1, 2))
    assert torch.allclose(Cs.float(), _ref(As, As, False, True), rtol=2.0 ** -10, atol=2e-3)
    # the fp32 FMA engine takes half operands too (it serves shapes the tensor engine cannot)
    Cf = ctx.defl_debug_gemm(A, B, ta, tb, engine=binding.ENGINE_SIMT, out_dtype=torch.float32)
    assert torch.allclose(Cf, ref, rtol=1e-4, atol=2e-3)


def test_bounded_wait_runs_out_and_is_reported(monkeypatch):
    """A device-side wait that nothing satisfies ends in a status bit and a normal return, not in a hang: one
    128 x 128 x 64 product (one CTA, one tile, one pipeline step) whose only pipeline step is never announced nor
    copied, with the wait limit at 2 ms. Nothing is in flight when the waits give up; the kernel frees its tensor
    memory and returns, the context stays usable and the next product is correct."""
    from paper_2609_21102_b200 import binding
    monkeypatch.setenv("DEFL_TC_WAIT_MS", "2")
    ctx = binding.Context(0)
    A, B = _mk(1, 128, 64, torch.bfloat16, 41), _mk(1, 128, 64, torch.bfloat16, 42)
    assert ctx.defl_device_wait_status() == 0
    ctx.defl_debug_gemm(A, B, False, True, engine=binding.ENGINE_TENSOR, out_dtype=torch.float32, withhold_first_step=True)
    assert ctx.defl_device_wait_status(clear=False) == binding.ST_DEVICE_WAIT
    assert ctx.defl_device_wait_status(clear=True) == binding.ST_DEVICE_WAIT      # sticky until cleared
    assert ctx.defl_device_wait_status() == 0
    C = ctx.defl_debug_gemm(A, B, False, True, engine=binding.ENGINE_TENSOR, out_dtype=torch.float32)
    assert torch.allclose(C, _ref(A, B, False, True), rtol=1e-4, atol=2e-3)
    assert ctx.defl_device_wait_status() == 0
    ctx.close()


def test_wait_limit_does_not_count_earlier_products(monkeypatch):
    """Products of one tile and a very deep K leave most of the chip free, so the next ones are resident while the first runs.
    The limit of their waits starts when their own work may: eight in a row, each shorter than the limit of 1.6 times
    one of them, finish without an event, and their results are the first one's."""
    from paper_2609_21102_b200 import binding
    K = 1 << 19
    A, B = _mk(1, 256, K, torch.bfloat16, 43), _mk(1, 256, K, torch.bfloat16, 44)
    free = binding.Context(0)
    product = lambda c: c.defl_debug_gemm(A, B, False, True, engine=binding.ENGINE_TENSOR, out_dtype=torch.float32)
    want = product(free)
    start, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    start.record()
    for _ in range(8):
        product(free)
    end.record()
    torch.cuda.synchronize()
    one = start.elapsed_time(end) / 8
    free.close()
    monkeypatch.setenv("DEFL_TC_WAIT_MS", str(int(1.6 * one) + 1))
    c = binding.Context(0)
    outs = [product(c) for _ in range(8)]
    assert c.defl_device_wait_status() == 0
    assert all(torch.equal(o, want) for o in outs)
    c.close()


@pytest.mark.parametrize("engine_name", ["simt", "tensor"])
@pytest.mark.parametrize("n,K", [(24, 24), (72, 200), (256, 64), (264, 264), (328, 1000), (640, 640)])
@pytest.mark.parametrize("dtype", [torch.float32, torch.float16])
def test_product_with_itself_is_the_full_product(ctx, engine_name, n, K, dtype):
    """A A^T given one buffer twice is computed by upper tiles and mirrored; given a copy as the second operand, in full. The
    tensor engine must give the same bits. The FMA engine may take another tile form, i.e. another order of the K terms:
    each of the two sums is within K rounding errors of 2^-24 on the sum of the magnitudes."""
    from paper_2609_21102_b200 import binding
    engine = binding.ENGINE_SIMT if engine_name == "simt" else binding.ENGINE_TENSOR
    A = _mk(2, n, K, dtype, 51)
    one = ctx.defl_debug_gemm(A, A, False, True, engine=engine, out_dtype=torch.float32)
    full = ctx.defl_debug_gemm(A, A.clone(), False, True, engine=engine, out_dtype=torch.float32)
    assert torch.equal(one, one.transpose(1, 2)) and torch.equal(full, full.transpose(1, 2))
    if engine_name == "tensor":
        assert torch.equal(one, full)
    else:
        bound = 2.0 * (K + 1) * 2.0 ** -24 * (A.double().abs() @ A.double().abs().transpose(1, 2))
        assert bool(((one.double() - full.double()).abs() <= bound).all())


@pytest.mark.parametrize("engine_name", ["simt", "tensor"])
@pytest.mark.parametrize("n", [40, 264, 520])
def test_polynomial_of_an_unsymmetric_matrix_is_computed_in_full(ctx, engine_name, n):
    """I + A + alpha A A^T for an A that is not symmetric, without exploit_symmetry: the product with itself alone does not
    make the result symmetric. (The second polynomial of a paired step meets this: its A is symmetric up to rounding.)"""
    from paper_2609_21102_b200 import binding
    engine = binding.ENGINE_SIMT if engine_name == "simt" else binding.ENGINE_TENSOR
    A = _mk(2, n, n, torch.float16, 52)
    C = ctx.defl_debug_gemm(A, A, False, True, engine=engine, out_dtype=torch.float32, alpha=0.125, polynomial=True)
    ref = torch.eye(n, device="cuda", dtype=torch.float64) + A.double() + 0.125 * (A.double() @ A.double().transpose(1, 2))
    bound = (n + 3) * 2.0 ** -23 * (1.0 + A.double().abs() + 0.125 * (A.double().abs() @ A.double().abs().transpose(1, 2)))
    assert bool(((C.double() - ref).abs() <= bound).all())


@pytest.mark.parametrize("width", [64, 96, 128, 160, 192, 224, 256])
def test_tensor_engine_every_tile_width(monkeypatch, width):
    """Every width that the tile rule can pick, forced (DEFL_TC_BN), on shapes that are multiples of none: K-major and MN-major
    operands (whose half tiles of 48, 80, 112 columns are not whole boxes), the symmetric store where the width does not
    divide the 256 rows of a tile (one operand given twice, and two operands that commute up to rounding: exactly symmetric
    in both cases), the transposed store, and the identity segment (a small deflated call)."""
    from paper_2609_21102_b200 import binding
    monkeypatch.setenv("DEFL_TC_BN", str(width))
    ctx = binding.Context(0)
    T = binding.ENGINE_TENSOR
    M, N, K = 712, 520, 328
    for ta, tb in ((False, True), (False, False), (True, True), (True, False)):
        A = _mk(2, K if ta else M, M if ta else K, torch.bfloat16, 61)
        B = _mk(2, N if tb else K, K if tb else N, torch.bfloat16, 62)
        ref = _ref(A, B, ta, tb)
        C = ctx.defl_debug_gemm(A, B, ta, tb, engine=T, out_dtype=torch.float32)
        assert torch.allclose(C, ref, rtol=1e-4, atol=4e-3)
        C = ctx.defl_debug_gemm(A, B, ta, tb, engine=T, out_dtype=torch.float32, transpose_out=True)
        assert torch.allclose(C, ref.transpose(1, 2), rtol=1e-4, atol=4e-3)
        A = A[:, :, :M - 8].contiguous() if ta else A[:, :M - 8].contiguous()      # (the symmetric shape: 704 rows)
        C = ctx.defl_debug_gemm(A, A, ta, not ta, engine=T, out_dtype=torch.float16, exploit_symmetry=True)
        ref = _ref(A, A, ta, not ta)
        assert torch.equal(C, C.transpose(1, 2)) and torch.allclose(C.float(), ref, rtol=2.0 ** -10, atol=4e-3)
    S = _mk(2, 456, 456, torch.float32, 63)
    S = (S + S.transpose(1, 2)).to(torch.float16) * 0.0625
    S2 = (S.float() @ S.float()).to(torch.float16)                # a polynomial in S: the two commute up to rounding
    S2 = torch.triu(S2) + torch.triu(S2, 1).transpose(1, 2)
    C = ctx.defl_debug_gemm(S, S2.contiguous(), False, True, engine=T, out_dtype=torch.float32, exploit_symmetry=True)
    ref = _ref(S, S2, False, True)
    err = 2.0 ** -11 * (S.double().abs() @ S2.double().abs()) * 2.0 + 1e-4     # S2's own rounding, in either order of the product
    assert torch.equal(C, C.transpose(1, 2)) and bool(((C.double() - ref.double()).abs() <= err).all())
    G = _mk(2, 264, 520, torch.bfloat16, 64)
    outs = [c.defl_polar_batched(G, 8, 8, 1, [list(binding.MUON_QUINTIC)] * 5, seed=4, gamma=1.01) for c in (ctx, binding.Context(0))]
    torch.cuda.synchronize()
    assert torch.equal(outs[0], outs[1])                         # a tile's width does not change the order of any sum
    ctx.close()
