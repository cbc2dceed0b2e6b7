"""Tensor-core kernels of the learned warm start (GPU required).

References are plain PyTorch CPU computations in FP64 of the same
BF16-rounded inputs; the tensor cores accumulate in FP32, so products agree
to a few FP32 ulps of the accumulated magnitude.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _bf16_pair(M, N, K, seed):
    import torch
    g = torch.Generator().manual_seed(seed)
    A = torch.randn(M, K, generator=g).to(torch.bfloat16)
    B = torch.randn(N, K, generator=g).to(torch.bfloat16)
    ref = A.double() @ B.double().T
    return A, B, ref


def _tol(ref, K):
    return 1e-5 * np.sqrt(K) * max(1.0, float(ref.abs().max()))


def test_gemm_layout_fields():
    """The descriptor's leading offset is the step between core matrices along
    K and the stride offset the step between 8-row groups (the reading of the
    no-swizzle K-major layout used by the kernel)."""
    import torch
    from paper_1406_2686_gb300 import nn
    A, B, ref = _bf16_pair(128, 32, 64, 1)
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    out = {}
    for swap in (0, 1):
        C = nn.gemm(A.cuda(), B.cuda(), layout=(128, 1024, swap), status=st)
        torch.cuda.synchronize()
        out[swap] = float((C.double().cpu() - ref).abs().max())
    assert int(st.item()) == 0
    print("layout errors (lbo field = K step, swapped):", out)
    assert out[0] < _tol(ref, 64)


@pytest.mark.parametrize("M,N,K", [(128, 32, 64), (256, 64, 128), (300, 48, 200), (1000, 128, 4096),
                                   (129, 16, 8), (4096, 100, 432), (384, 256, 320), (700, 200, 1000),
                                   (512, 640, 264), (130, 129, 72)])
def test_gemm_matches_fp64(M, N, K):
    import torch
    from paper_1406_2686_gb300 import nn
    A, B, ref = _bf16_pair(M, N, K, M + N + K)
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    C = nn.gemm(A.cuda(), B.cuda(), status=st)
    torch.cuda.synchronize()
    assert int(st.item()) == 0
    err = float((C.double().cpu() - ref).abs().max())
    assert err < _tol(ref, K), err


@pytest.mark.parametrize("K,k_split", [(1000, 256), (4096, 1024), (200, 64)])
def test_gemm_splitk_slices_sum_to_product(K, k_split):
    """The split-K form: slice z reduces K in [z k_split, (z + 1) k_split) into
    its own C slice (the last slice ragged, zero-filled beyond K); the slices
    sum to A B^T, and each slice equals the product of its K range."""
    import torch
    from paper_1406_2686_gb300 import nn
    M, N = 260, 96
    A, B, ref = _bf16_pair(M, N, K, K + k_split)
    splits = (K + k_split - 1) // k_split
    parts = torch.full((splits, M, N), 7.0, dtype=torch.float32, device="cuda")
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    lb = nn.L()
    Ad, Bd = A.cuda(), B.cuda()  # kept alive until the kernel has run
    nn._check(lb.vefd_nn_gemm_bf16_splitk(Ad.data_ptr(), K, Bd.data_ptr(), K, parts.data_ptr(), N, M, N, K, k_split,
                                          M * N, st.data_ptr(), nn._stream()), "splitk")
    torch.cuda.synchronize()
    assert int(st.item()) == 0
    got = parts.double().cpu()
    assert float((got.sum(0) - ref).abs().max()) < _tol(ref, K)
    for z in range(splits):
        k0, k1 = z * k_split, min(K, (z + 1) * k_split)
        sub = A[:, k0:k1].double() @ B[:, k0:k1].double().T
        assert float((got[z] - sub).abs().max()) < _tol(sub, k1 - k0), z


def test_gemm_accumulate_and_strides():
    """C += A B^T into a strided view keeps the old values and the untouched columns."""
    import torch
    from paper_1406_2686_gb300 import nn
    A, B, ref = _bf16_pair(200, 40, 96, 7)
    Cbig = torch.full((200, 64), 2.5, dtype=torch.float32, device="cuda")
    C = Cbig[:, 8:48]
    nn.gemm(A.cuda(), B.cuda(), C=C, accumulate=True)
    torch.cuda.synchronize()
    got = Cbig.double().cpu()
    assert float((got[:, 8:48] - (ref + 2.5)).abs().max()) < _tol(ref, 96)
    assert torch.all(got[:, :8] == 2.5) and torch.all(got[:, 48:] == 2.5)


def test_gemm_rejects_bad_arguments():
    import torch
    from paper_1406_2686_gb300 import nn
    A = torch.zeros(128, 12, dtype=torch.bfloat16, device="cuda")  # K not a multiple of 8
    B = torch.zeros(32, 12, dtype=torch.bfloat16, device="cuda")
    with pytest.raises(nn.NNError):
        nn.gemm(A, B)
    A = torch.zeros(128, 64, dtype=torch.bfloat16, device="cuda")
    B = torch.zeros(32, 64, dtype=torch.bfloat16, device="cuda")
    with pytest.raises(nn.NNError):
        nn.gemm(A, B, layout=(4096, 4096, 0))  # would leave the staged tile


# --- convolution layers and the network against PyTorch CPU autograd (FP64) ----

def _torch_weight(lay):
    """Our w[o][((dz*3+dy)*3+dx)*Cin + c] (BF16-rounded) as torch [Cout, Cin, 3, 3, 3]."""
    import torch
    w = lay.w.cpu().to(torch.bfloat16).double()
    return w.view(lay.cout, 3, 3, 3, lay.cin).permute(0, 4, 1, 2, 3).contiguous()


def _ncdhw(x):
    return x.permute(0, 4, 1, 2, 3)


def _rel(a, b):
    import torch
    return float(torch.linalg.norm((a - b).flatten()) / max(1e-30, float(torch.linalg.norm(b.flatten()))))


@pytest.mark.parametrize("cin,cout,stride,relu,shape", [(5, 16, 1, True, (1, 8, 8, 16)), (16, 32, 2, True, (2, 8, 16, 8)),
                                                        (24, 8, 1, False, (1, 16, 8, 8))])
def test_conv_layer_matches_torch(cin, cout, stride, relu, shape):
    """Forward values and the gradients of input, weights and bias of one
    convolution layer agree with FP64 autograd of the same BF16-rounded
    weights (the GEMM operands are BF16: a few 1e-3 relative)."""
    import torch
    import torch.nn.functional as F
    from paper_1406_2686_gb300 import nn
    g = torch.Generator().manual_seed(cin + cout)
    lay = nn.Conv3d(cin, cout, stride, relu, gen=g)
    lay.b.copy_(torch.randn(cout, generator=g).cuda() * 0.1)
    x = torch.randn(*shape, cin, generator=g)
    y = lay.forward(x.cuda().contiguous())
    dy = torch.randn(*y.shape, generator=g)
    dx = lay.backward(dy.cuda())
    torch.cuda.synchronize()
    xr = _ncdhw(x.to(torch.bfloat16).double()).requires_grad_(True)
    wr = _torch_weight(lay).requires_grad_(True)
    br = lay.b.cpu().double().requires_grad_(True)
    yr = F.conv3d(xr, wr, br, stride=stride, padding=1)
    if relu:
        yr = F.relu(yr)
    yr.backward(_ncdhw(dy.double()))
    assert _rel(_ncdhw(y.cpu().double()), yr.detach()) < 1e-2
    assert _rel(_ncdhw(dx.cpu().double()), xr.grad) < 2e-2
    dwr = wr.grad.permute(0, 2, 3, 4, 1).reshape(cout, -1)
    assert _rel(lay.dw.cpu().double(), dwr) < 2e-2
    assert _rel(lay.db.cpu().double(), br.grad) < 1e-3
    assert int(lay.status.item()) == 0


@pytest.mark.parametrize("cin,cout,stride,shape", [
    (8, 8, 1, (1, 1, 1, 8)), (8, 16, 2, (1, 5, 3, 16)), (3, 24, 1, (2, 3, 5, 8)), (24, 40, 1, (1, 7, 9, 8)),
    (48, 16, 1, (1, 6, 10, 24)), (16, 264, 1, (1, 2, 3, 8)), (232, 80, 1, (1, 4, 4, 8)), (40, 152, 2, (2, 7, 6, 16)),
    (16, 32, 2, (1, 2, 1, 16)), (64, 256, 1, (1, 3, 3, 8)), (48, 16, 1, (1, 20, 18, 24)), (16, 32, 2, (1, 20, 36, 32)),
    (112, 16, 2, (1, 4, 4, 16)), (264, 8, 1, (1, 2, 2, 8)), (16, 296, 2, (1, 3, 2, 16)), (152, 152, 1, (1, 8, 8, 8))])
def test_conv_products(cin, cout, stride, shape):
    """The products at the edges of their tiles (one voxel row, ragged rows and
    channel slabs, several column tiles and channel blocks, odd sizes at stride 2) against
    FP64 of the BF16 operands they multiply: only FP32 accumulation is left,
    over K terms an error below sqrt(K) 2^-23 of the terms' size; 1e-5 sqrt(K)
    of the largest value is the bound of the other products here."""
    import torch
    import torch.nn.functional as F
    from paper_1406_2686_gb300 import nn
    g = torch.Generator().manual_seed(cin * 7 + cout)
    lay = nn.Conv3d(cin, cout, stride, False, gen=g)
    x = torch.randn(*shape, cin, generator=g)
    y = lay.forward(x.cuda().contiguous())
    dy = torch.randn(*y.shape, generator=g).to(torch.bfloat16).float()
    dx = lay.backward(dy.cuda())
    torch.cuda.synchronize()
    assert int(lay.status.item()) == 0
    xr = _ncdhw(x.to(torch.bfloat16).double()).requires_grad_(True)
    wr = _torch_weight(lay).requires_grad_(True)
    yr = F.conv3d(xr, wr, None, stride=stride, padding=1)
    yr.backward(_ncdhw(dy.double()))
    V = y.numel() // cout
    for got, ref, K in ((_ncdhw(y.cpu().double()), yr.detach(), 27 * cin), (_ncdhw(dx.cpu().double()), xr.grad, 27 * cout),
                        (lay.dw.cpu().double(), wr.grad.permute(0, 2, 3, 4, 1).reshape(cout, -1), V),
                        (lay.db.cpu().double(), dy.double().sum((0, 1, 2, 3)), V)):
        assert float((got - ref).abs().max()) < _tol(ref, K)


@pytest.mark.parametrize("channels", [(8, 16, 32, 64), (8, 16, 24, 40)])
def test_unet_gradients_match_torch(channels):
    """The whole U-Net (forward, MSE loss, backward through every layer, skip
    and upsampling) against FP64 autograd of the same weights, for the
    doubling channel plan and an uneven one."""
    import torch
    import torch.nn.functional as F
    from paper_1406_2686_gb300 import nn
    net = nn.UNet(5, 8, seed=3, channels=channels)
    g = torch.Generator().manual_seed(5)
    for lay in net.layers:
        lay.b.copy_(torch.randn(lay.cout, generator=g).cuda() * 0.05)
    x = torch.randn(1, 16, 16, 16, 5, generator=g)
    t = torch.randn(1, 16, 16, 16, 8, generator=g)
    out = net.forward(x.cuda().contiguous())
    loss_parts, grad = nn.mse(out, t.cuda().contiguous())
    net.backward(grad)
    torch.cuda.synchronize()
    loss = float(loss_parts.sum()) / out.numel()

    W = {id(l): _torch_weight(l).requires_grad_(True) for l in net.layers}
    Bv = {id(l): l.b.cpu().double().requires_grad_(True) for l in net.layers}

    def run(layers, h):
        for l in layers:
            h = F.conv3d(h, W[id(l)], Bv[id(l)], stride=l.stride, padding=1)
            if l.relu:
                h = F.relu(h)
        return h

    up = lambda h: F.interpolate(h, scale_factor=2, mode="nearest")
    xr = _ncdhw(x.double())
    s0 = run(net.e0, xr)
    s1 = run(net.e1, s0)
    s2 = run(net.e2, s1)
    s3 = run(net.e3, s2)
    u2 = run(net.d2, torch.cat([up(s3), s2], 1))
    u1 = run(net.d1, torch.cat([up(u2), s1], 1))
    o = run(net.d0, torch.cat([up(u1), s0], 1))
    lr = ((o - _ncdhw(t.double())) ** 2).mean()
    lr.backward()
    assert abs(loss / float(lr.detach()) - 1) < 2e-2
    assert _rel(_ncdhw(out.cpu().double()), o.detach()) < 3e-2
    # every GEMM rounds its operands (activations, gradients) to BF16, so the
    # error grows along the backward chain: direction and size are compared
    for l in net.layers:
        dwr = W[id(l)].grad.permute(0, 2, 3, 4, 1).reshape(l.cout, -1)
        for a, r in ((l.dw.cpu().double(), dwr), (l.db.cpu().double(), Bv[id(l)].grad)):
            cos = float((a * r).sum() / (torch.linalg.norm(a) * torch.linalg.norm(r)))
            assert cos > 0.995 and abs(float(torch.linalg.norm(a) / torch.linalg.norm(r)) - 1) < 0.05, (l.cout, cos)
            assert _rel(a, r) < 0.1
    assert net.status() == 0


def _conv_fp64(x, w, dy, stride):
    """y, dx, dw of a convolution in FP64 tap by tap: x [B][D][H][W][C], w
    [Cout][27][C], dy as y."""
    import torch
    xp = torch.nn.functional.pad(x, (0, 0, 1, 1, 1, 1, 1, 1))
    B, Do, Ho, Wo, O = dy.shape
    y, dw, dxp = torch.zeros_like(dy), torch.zeros_like(w), torch.zeros_like(xp)
    for t in range(27):
        at = (slice(None), *(slice(o, o + stride * (n - 1) + 1, stride) for o, n in
                             zip((t // 9, t // 3 % 3, t % 3), (Do, Ho, Wo))))
        y += xp[at] @ w[:, t].T
        dw[:, t] = dy.reshape(-1, O).T @ xp[at].reshape(-1, x.shape[-1])
        dxp[at] += dy @ w[:, t]
    return y, dxp[:, 1:-1, 1:-1, 1:-1], dw


# what the plan for 152 SMs takes each shape through: k_conv's 128-row products
# and their epilogue with rows beyond the grid, 1, 2 and 4 planes a tile, two to
# three items a block over two and over one halo buffer and over two and one
# accumulator sets, and 3 to 18 tiles a block in k_conv_dw's ring of 2 to 4
@pytest.mark.parametrize("cin,cout,stride,shape", [
    (16, 16, 1, (1, 61, 58, 64)),   # 4 planes
    (8, 16, 1, (1, 66, 58, 60)),    # 4 planes, odd slabs
    (48, 16, 1, (1, 41, 52, 40)),   # 2 planes, three items
    (112, 32, 1, (1, 36, 44, 60)),  # 2 planes, one halo buffer; gradient of 112 columns
    (112, 32, 1, (1, 35, 40, 44)),  # 4 planes, one halo buffer; gradient on one accumulator set
    (40, 24, 2, (1, 60, 44, 72)),   # odd slabs; adjoint on one accumulator set; ring of 2
    (16, 32, 2, (1, 92, 84, 92)),   # 4 planes of 8 rows
    (32, 16, 2, (2, 66, 64, 60)),   # two grids
    (232, 80, 1, (1, 18, 28, 36)),  # 98 weight chunks an item; gradient in three column tiles of 4 planes
])
def test_conv_products_over_many_tiles(cin, cout, stride, shape):
    """The products where a block walks several tiles, against FP64 of the BF16
    operands; the bound is that of test_conv_products."""
    import torch
    from paper_1406_2686_gb300 import nn
    g = torch.Generator().manual_seed(cin + 3 * cout + stride)
    lay = nn.Conv3d(cin, cout, stride, False, gen=g)
    x = torch.randn(*shape, cin, generator=g).cuda()
    xb = torch.empty(x[..., 0].numel(), nn.round8(cin), dtype=torch.bfloat16, device="cuda")
    yb = torch.full(lay.out_shape(x.shape), float("nan"), dtype=torch.bfloat16, device="cuda")
    y = lay._forward(x, xb, x.shape, yb, nn._stream())
    assert torch.equal(yb, y.to(torch.bfloat16))  # the copy that the next layer reads
    dy = torch.randn(*y.shape, generator=g).to(torch.bfloat16).float().cuda()
    dx = lay.backward(dy)
    assert int(lay.status.item()) == 0
    w = lay.w.to(torch.bfloat16).double().view(cout, 27, cin)
    yr, dxr, dwr = _conv_fp64(x.to(torch.bfloat16).double(), w, dy.double(), stride)
    V = y.numel() // cout
    for got, ref, K in ((y, yr, 27 * cin), (dx, dxr, 27 * cout), (lay.dw.view(cout, 27, cin), dwr, V),
                        (lay.db, dy.double().sum((0, 1, 2, 3)), V)):
        assert float((got.double() - ref).abs().max()) < _tol(ref, K)


@pytest.mark.parametrize("cin,cout,stride,shape,bits", [
    (16, 16, 1, (1, 66, 60, 44), True), (24, 16, 1, (1, 20, 18, 24), True), (232, 80, 1, (1, 8, 8, 8), True),
    (40, 24, 2, (2, 9, 12, 16), True), (256, 32, 1, (1, 4, 8, 8), True), (96, 16, 2, (1, 8, 8, 16), True),
    (12, 16, 1, (1, 8, 8, 16), False), (264, 16, 1, (1, 4, 8, 8), False), (104, 16, 2, (1, 8, 8, 16), False)])
def test_conv_layer_agrees_with_the_im2col_route(cin, cout, stride, shape, bits):
    """The layer against the exported im2col matrices, GEMMs and element kernels.
    The forward bits are the same where both sum in the same order (one block
    of a multiple of 8 channels); what is left is FP32 accumulation on both
    sides, twice the bound of one."""
    import torch
    from paper_1406_2686_gb300 import nn
    g = torch.Generator().manual_seed(cin + cout)
    lay = nn.Conv3d(cin, cout, stride, True, gen=g)
    lay.b.copy_(torch.randn(cout, generator=g).cuda() * 0.1)
    x = torch.randn(*shape, cin, generator=g).cuda()
    y = lay.forward(x)
    V, K27, Kp = y.numel() // cout, 27 * cin, nn.round8(27 * cin)
    dy = torch.randn(*y.shape, generator=g).cuda()
    lb, s, st = nn.L(), nn._stream(), torch.zeros(1, dtype=torch.int32, device="cuda")

    def empty(*size, dtype=torch.bfloat16):
        return torch.empty(*size, dtype=dtype, device="cuda")

    def call(name, *args):
        nn._check(getattr(lb, "vefd_nn_" + name)(*[nn._p(a) if torch.is_tensor(a) else a for a in args], s), name)

    col, colT, wb, wbT = empty(V, Kp), empty(Kp, V), empty(cout, Kp), empty(Kp, cout)
    call("im2col3d", x, *shape, cin, stride, Kp, col, colT)
    call("pack_weights", lay.w, cout, K27, Kp, wb, wbT)
    r = nn.gemm(col, wb, status=st)
    call("bias_act", r, lay.b, V, cout, 1)
    r = r.view(y.shape)
    if bits:
        assert torch.equal(y, r)
    assert float((y - r).abs().max()) < 2 * _tol(r, K27)

    # the gradients for one forward output: the mask is then the same
    lay._saved = (x.shape, lay._saved[1], r)
    dx = lay.backward(dy)
    f32 = torch.float32
    gr, gb, gbT = empty(V, cout, dtype=f32), empty(V, cout), empty(cout, V)
    call("act_backward", dy, r, V, cout, 1, gr, gb, gbT)
    db, dw = empty(cout, dtype=f32), empty(cout, K27, dtype=f32)
    call("colsum", gr, V, cout, empty(lb.vefd_nn_colsum_scratch(V, cout), dtype=f32), db, 0)
    ks = 64 * ((V + 255) // 256)
    splits = (V + ks - 1) // ks
    parts = empty(splits, Kp, cout, dtype=f32)
    nn._check(lb.vefd_nn_gemm_bf16_splitk(colT.data_ptr(), V, gbT.data_ptr(), V, parts.data_ptr(), cout, Kp, cout, V, ks,
                                          Kp * cout, st.data_ptr(), s), "splitk")
    call("splitk_reduce_t", parts, splits, Kp * cout, Kp, cout, K27, dw, 0)
    dcol, dxr = nn.gemm(gb, wbT, status=st), empty(*x.shape, dtype=f32)
    call("col2im3d", dcol, *shape, cin, stride, Kp, dxr)
    assert int(st.item()) == 0 and int(lay.status.item()) == 0
    for a, b, K in ((dx, dxr, 27 * cout), (lay.dw, dw, V), (lay.db, db, V)):
        assert float((a - b).abs().max()) < 2 * _tol(b, K)


def test_upsample_and_concat():
    """The FP32 forms of what the network's fused pass does: copies, so exact."""
    import torch
    from paper_1406_2686_gb300 import nn
    g = torch.Generator().manual_seed(2)
    u, sk = (torch.randn(2, d, d + 1, d + 2, c, generator=g).cuda() for d, c in ((3, 16), (3, 8)))
    up = nn.upsample2(u)
    for k in (1, 2, 3):
        u = u.repeat_interleave(2, dim=k)
        sk = sk.repeat_interleave(2, dim=k)
    assert torch.equal(up, u)
    assert torch.equal(nn.concat(up, sk.contiguous()), torch.cat([u, sk], dim=-1))
