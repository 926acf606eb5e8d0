"""Kernels at the edges of their tiles and of their dispatch rules, against
plain FP64 PyTorch (the layers) or the general path (the traced ones).

Tolerances: a BF16 output is rounded once from an FP32 value; BF16 has 8
significant bits, so the error is at most 2^-8 of each element (1 + 2^-8 lies
half way between two BF16 numbers); the FP32 sums before it (at most 2304
products here) add below 1e-5 of the result's size.  So BF16 outputs are held
to 2^-8 + 1e-5 in the 2-norm.
"""
import ctypes as C
import math

import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
BF = torch.bfloat16
BF_TOL = 2.0 ** -8 + 1e-5


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()


def ops():
    from paper_2408_15583_gb300.learned import Ops
    return Ops(DEV)


def rel(a, b):
    a, b = a.double(), b.double()
    return float((a - b).norm() / b.norm().clamp(min=1e-30))


def gen(seed):
    return torch.Generator(device=DEV).manual_seed(seed)


def rnd(g, *s):
    return torch.randn(*s, generator=g, device=DEV)


# ---- the streaming contraction ------------------------------------------------

# rows: one, a warp's 32 and its neighbours, a tile's 128 and its neighbours,
# more tiles than resident CTAs; columns: inside one slab, ragged slabs, every
# column tile, two column tiles; K: below one block, ragged, several blocks
@pytest.mark.parametrize("mode", ["plain", "residual", "gelu", "dgelu"])
@pytest.mark.parametrize("M,N,K", [(1, 32, 32), (31, 8, 16), (33, 40, 64), (127, 64, 72),
                                   (129, 136, 128), (128, 128, 576), (160, 256, 64),
                                   (90_000, 32, 128), (60_001, 96, 32)])
def test_streaming_contraction(M, N, K, mode):
    o, g = ops(), gen(M + N + K)
    A, B = rnd(g, M, K).to(BF), (rnd(g, N, K) / math.sqrt(K)).to(BF)
    bias = rnd(g, N)
    X = rnd(g, M, N + 8).to(BF)                       # a wider row than the output's
    out = torch.full((M, N + 16), 7.0, dtype=BF, device=DEV)
    Z = torch.full((M, N + 8), 7.0, dtype=BF, device=DEV)
    ref = A.double() @ B.double().T
    kw = {}
    if mode == "plain":
        kw = dict(bias=bias)
        want = ref + bias.double()
    elif mode == "residual":
        kw = dict(bias=bias, R=X, ldr=N + 8)
        want = ref + bias.double() + X[:, :N].double()
    elif mode == "gelu":
        kw = dict(bias=bias, Z=Z, ldz=N + 8, gelu=True)
        pre = ref + bias.double()
        want = torch.nn.functional.gelu(pre)
    else:
        kw = dict(Z=X, ldz=N + 8, dgelu=True)
        z = X[:, :N].double()
        want = ref * (0.5 * (1 + torch.erf(z / math.sqrt(2))) +
                      z * torch.exp(-0.5 * z * z) / math.sqrt(2 * math.pi))
    o.gemm(M, N, K, A, K, 1, B, 1, K, out, N + 16, **kw)
    assert rel(out[:, :N], want) < BF_TOL
    assert bool((out[:, N:] == 7.0).all())            # nothing past the row's columns
    if mode == "gelu":
        assert rel(Z[:, :N], pre) < BF_TOL
        assert bool((Z[:, N:] == 7.0).all())
    from paper_2408_15583_gb300 import api
    api.stream_check()


@pytest.mark.parametrize("mode", ["plain", "residual", "gelu"])
def test_streaming_contraction_gives_up_and_recovers(mode):
    """With a limit of zero polls no wait of the main loop succeeds: nothing is
    stored, the status word says so once, and the next call computes."""
    from paper_2408_15583_gb300 import _lib
    lib = _lib.load()
    o, g = ops(), gen(3)
    M, N, K = 5000, 128, 128
    A, B = rnd(g, M, K).to(BF), rnd(g, N, K).to(BF)
    R = rnd(g, M, N).to(BF)
    Z = torch.zeros(M, N, dtype=BF, device=DEV)
    kw = dict(residual=dict(R=R, ldr=N), gelu=dict(Z=Z, ldz=N, gelu=True)).get(mode, {})
    stream = C.c_void_p(torch.cuda.current_stream().cuda_stream)
    try:
        assert lib.pe_nn_set_wait_limit(0) == 0
        out = torch.zeros(M, N, dtype=BF, device=DEV)
        o.gemm(M, N, K, A, K, 1, B, 1, K, out, N, **kw)
        assert lib.pe_stream_check(stream) == 4       # PE_ETIMEOUT
        assert torch.count_nonzero(out) == 0 and torch.count_nonzero(Z) == 0
        assert lib.pe_stream_check(stream) == 0
    finally:
        lib.pe_nn_set_wait_limit(-1)
    o.gemm(M, N, K, A, K, 1, B, 1, K, out, N, **kw)
    assert lib.pe_stream_check(stream) == 0
    pre = A.double() @ B.double().T + (R.double() if mode == "residual" else 0.0)
    assert rel(out, torch.nn.functional.gelu(pre) if mode == "gelu" else pre) < BF_TOL


# with few polls a wait deep in the loop may fail, in any role, while others have
# copies or products in flight: the call says so or is whole, and the next computes
@pytest.mark.parametrize("polls", [1, 2, 5])
@pytest.mark.parametrize("mode", ["plain", "residual", "gelu", "wgrad"])
def test_contraction_recovers_whichever_wait_gives_up(mode, polls):
    from paper_2408_15583_gb300 import _lib
    lib = _lib.load()
    o, g = ops(), gen(polls)
    M, N, K = 90_000, 128, 320
    A, B = rnd(g, M, K).to(BF), rnd(g, N, K).to(BF)
    R, Z = rnd(g, M, N).to(BF), torch.empty(M, N, dtype=BF, device=DEV)
    kw = dict(residual=dict(R=R, ldr=N), gelu=dict(Z=Z, ldz=N, gelu=True)).get(mode, {})
    stream = C.c_void_p(torch.cuda.current_stream().cuda_stream)
    out = torch.empty(M, N, dtype=BF, device=DEV)
    dW, db = torch.empty(N, K, device=DEV), torch.empty(N, device=DEV)
    ws = torch.empty(lib.pe_nn_linear_wgrad_workspace(M, N, K), dtype=torch.uint8, device=DEV)
    ptr = lambda t: C.c_void_p(t.data_ptr())

    def call():
        if mode == "wgrad":
            assert lib.pe_nn_linear_wgrad(ptr(R), N, ptr(A), K, M, N, K, ptr(dW), ptr(db), ptr(ws),
                                          ws.numel(), stream) == 0
        else:
            o.gemm(M, N, K, A, K, 1, B, 1, K, out, N, **kw)
        return lib.pe_stream_check(stream), (dW if mode == "wgrad" else out).clone()

    status, want = call()
    assert status == 0
    for _ in range(3):
        try:
            assert lib.pe_nn_set_wait_limit(polls) == 0
            status, got = call()
        finally:
            lib.pe_nn_set_wait_limit(-1)
        assert status in (0, 4)                       # PE_OK or PE_ETIMEOUT
        assert status == 4 or torch.equal(got, want)
        status, got = call()
        assert status == 0 and torch.equal(got, want)


# ---- depthwise 7x7 --------------------------------------------------------------

# images smaller than the stencil, ragged rows and columns, odd pair counts and
# more than one chunk of channel pairs, and enough positions for four rows per
# thread; the weight gradient's FP32 sums (over at most 2 * 96 * 200 pixels, in
# runs of a few hundred) err below 1e-5
@pytest.mark.parametrize("B,H,W,C", [(1, 1, 1, 2), (2, 3, 5, 6), (1, 9, 17, 32), (2, 12, 33, 40),
                                     (1, 7, 70, 130), (2, 96, 200, 64), (3, 130, 131, 256)])
def test_depthwise(B, H, W, C):
    o, g = ops(), gen(B + H + W + C)
    x, dy = rnd(g, B, H, W, C).to(BF), rnd(g, B, H, W, C).to(BF)
    w, b = rnd(g, 7, 7, C) / 7, rnd(g, C)
    P = B * H * W
    y, dx = torch.empty(P, C, dtype=BF, device=DEV), torch.empty(P, C, dtype=BF, device=DEV)
    dw, db = torch.empty(7, 7, C, device=DEV), torch.empty(C, device=DEV)
    o.dw(x, w, b, B, H, W, C, y)
    o.dw_bwd(x, dy, w, B, H, W, C, dx, dw, db)
    pad = lambda t: torch.nn.functional.pad(t.double(), (0, 0, 3, 3, 3, 3))
    xp, gp = pad(x), pad(dy)
    ry = b.double().expand(B, H, W, C).clone()
    rx, rw = torch.zeros_like(ry), torch.empty(7, 7, C, dtype=torch.float64, device=DEV)
    for i in range(7):
        for j in range(7):
            win = xp[:, i:i + H, j:j + W]
            ry += w[i, j].double() * win
            rx += w[6 - i, 6 - j].double() * gp[:, i:i + H, j:j + W]
            rw[i, j] = (win * dy.double()).sum((0, 1, 2))
    assert rel(y.view(B, H, W, C), ry) < BF_TOL
    assert rel(dx.view(B, H, W, C), rx) < BF_TOL
    assert rel(dw, rw) < 1e-5
    assert rel(db, dy.double().sum((0, 1, 2))) < 1e-5


# an infinity or NaN of X reaches exactly the taps that read it: one per channel
# pair, near each side of images whose rows are and are not whole groups of eight
@pytest.mark.parametrize("H,W", [(9, 17), (4, 5), (7, 64), (40, 130), (2, 16)])
@pytest.mark.parametrize("value", [math.inf, math.nan])
def test_depthwise_weight_gradient_of_infinities(H, W, value):
    o, g, B, C = ops(), gen(H + W), 2, 64
    x, dy = rnd(g, B, H, W, C).to(BF), rnd(g, B, H, W, C).to(BF)
    spots = [(y, x_) for y in (0, 1, 2, H - 1, H - 2, H // 2) for x_ in (0, 2, W - 1, W - 2, W // 2)
             if 0 <= y < H and 0 <= x_ < W][:C // 2]
    for k, (y, x_) in enumerate(spots):
        x[k % B, y, x_, 2 * k] = value
    w = rnd(g, 7, 7, C)
    dx = torch.empty(B * H * W, C, dtype=BF, device=DEV)
    dw, db = torch.empty(7, 7, C, device=DEV), torch.empty(C, device=DEV)
    o.dw_bwd(x, dy, w, B, H, W, C, dx, dw, db)
    xp = torch.nn.functional.pad(x.double(), (0, 0, 3, 3, 3, 3))
    want = torch.stack([(xp[:, i:i + H, j:j + W] * dy.double()).sum((0, 1, 2))
                        for i in range(7) for j in range(7)]).view(7, 7, C)
    assert torch.equal(dw.isfinite(), want.isfinite())
    ok = want.isfinite()
    assert bool((~ok).any()) and rel(dw[ok], want[ok]) < 1e-5
    assert rel(db, dy.double().sum((0, 1, 2))) < 1e-5


# the split of the weight gradient: positions added side by side (64 for two channels
# to two for 64 and more), stretches of 8 to 64 pixels, more blocks for 128 channels and up
@pytest.mark.parametrize("B,H,W,C", [(1, 64, 64, 8), (1, 3, 200, 2), (2, 33, 9, 6), (3, 40, 130, 12),
                                     (4, 64, 64, 32), (40, 32, 32, 128), (34, 32, 17, 256)])
def test_depthwise_weight_gradient_split(B, H, W, C):
    o, g = ops(), gen(B + H + W + C)
    x, dy = rnd(g, B, H, W, C).to(BF), rnd(g, B, H, W, C).to(BF)
    w = rnd(g, 7, 7, C)
    dx = torch.empty(B * H * W, C, dtype=BF, device=DEV)
    dw, db = torch.empty(7, 7, C, device=DEV), torch.empty(C, device=DEV)
    o.dw_bwd(x, dy, w, B, H, W, C, dx, dw, db)
    xp = torch.nn.functional.pad(x.double(), (0, 0, 3, 3, 3, 3))
    want = torch.stack([(xp[:, i:i + H, j:j + W] * dy.double()).sum((0, 1, 2))
                        for i in range(7) for j in range(7)]).view(7, 7, C)
    assert rel(dw, want) < 1e-5
    assert rel(db, dy.double().sum((0, 1, 2))) < 1e-5


# ---- LayerNorm ------------------------------------------------------------------

# one pixel, a block's 64 and its neighbours, more pixels than resident blocks;
# every channel count of the four-threads-per-pixel kernels and one beside them
@pytest.mark.parametrize("C", [32, 40, 64, 128, 256])
@pytest.mark.parametrize("P", [1, 63, 65, 100_003])
def test_layernorm(P, C):
    o, g = ops(), gen(P + C)
    x, dy = (rnd(g, P, C) + 0.5).to(BF), rnd(g, P, C).to(BF)
    gam, bet = rnd(g, C), rnd(g, C)
    y, dx = torch.empty(P, C, dtype=BF, device=DEV), torch.empty(P, C, dtype=BF, device=DEV)
    mean, rstd = torch.empty(P, device=DEV), torch.empty(P, device=DEV)
    dg, db = torch.empty(C, device=DEV), torch.empty(C, device=DEV)
    o.ln(x, gam, bet, P, C, y, mean, rstd)
    o.ln_bwd(dy, x, gam, mean, rstd, P, C, dx, dg, db)
    xd = x.double().requires_grad_(True)
    gd, bd = gam.double().requires_grad_(True), bet.double().requires_grad_(True)
    ref = torch.nn.functional.layer_norm(xd, (C,), gd, bd, 1e-6)
    ref.backward(dy.double())
    assert rel(y, ref.detach()) < BF_TOL
    assert rel(mean, x.double().mean(1)) < 1e-5
    assert rel(dx, xd.grad) < BF_TOL
    assert rel(dg, gd.grad) < 1e-5 and rel(db, bd.grad) < 1e-5


# ---- weight gradients -------------------------------------------------------------

# pixels below a block, ragged blocks, one and many splits; widths below a box,
# either operand the wider one, several accumulators, several tiles each way;
# FP32 sums over P products err below 1e-5 of the result
@pytest.mark.parametrize("N,K", [(8, 8), (32, 128), (128, 32), (64, 256), (136, 40), (128, 576),
                                 (264, 520)])
@pytest.mark.parametrize("P", [16, 63, 200, 70_001])
def test_linear_weight_gradient(P, N, K):
    from paper_2408_15583_gb300 import _lib, api
    lib = _lib.load()
    g = gen(P + N + K)
    dy, x = rnd(g, P, N).to(BF), rnd(g, P, K + 8).to(BF)
    dW, db = torch.full((N, K), 7.0, device=DEV), torch.full((N,), 7.0, device=DEV)
    nb = lib.pe_nn_linear_wgrad_workspace(P, N, K)
    ws = torch.empty(nb, dtype=torch.uint8, device=DEV)
    ptr = lambda t: C.c_void_p(t.data_ptr())
    stream = C.c_void_p(torch.cuda.current_stream().cuda_stream)
    call = lambda: lib.pe_nn_linear_wgrad(ptr(dy), N, ptr(x), K + 8, P, N, K, ptr(dW), ptr(db),
                                          ptr(ws), nb, stream)
    try:                                # its bounded waits give up and say so
        assert lib.pe_nn_set_wait_limit(0) == 0
        assert call() == 0 and lib.pe_stream_check(stream) == 4
    finally:
        lib.pe_nn_set_wait_limit(-1)
    assert call() == 0
    api.stream_check()
    assert rel(dW, dy.double().T @ x[:, :K].double()) < 1e-5
    assert rel(db, dy.double().sum(0)) < 1e-5


# the bias gradient of long stretches: dY = 1 at 64 pixels of every 4096, else 2^-22,
# half an ulp of what a plain chain of sums then holds (it drops nearly all of
# them: 78 to 144 ulps).  With the errors kept, what is left to round: each
# thread's sum, two shuffles, three warps, the splits by eights and their eight sums
@pytest.mark.parametrize("N,K", [(1024, 256), (512, 576), (128, 1152)])
def test_bias_gradient_of_long_stretches(N, K):
    o, g, P = ops(), gen(N), 131072
    dy = torch.full((P, N), 2.0 ** -22, dtype=BF, device=DEV)
    dy.view(P // 4096, 4096, N)[:, :64] = 1.0
    x, W = rnd(g, P, K).to(BF), rnd(g, N, K).to(BF)
    dW, db = torch.empty(N, K, device=DEV), torch.empty(N, device=DEV)
    o.linear_bwd(dy, x, K, W, None, 0, dW, db, need_dx=False)
    want = float(dy[:, 0].double().sum())
    splits = o.lib.pe_nn_linear_wgrad_workspace(P, N, K) // (4 * (N * K + N))   # at most
    steps = 1 + 2 + 3 + -(-splits // 8) + 8
    assert float((db.double() - want).abs().max()) <= steps * 2.0 ** -24 * want

# an infinite or NaN dY reaches its own bias and weights alone, as infinity or NaN
@pytest.mark.parametrize("N,K", [(256, 64), (64, 256)])
def test_bias_gradient_of_infinities(N, K):
    o, g, P = ops(), gen(N), 5000
    dy, x = rnd(g, P, N).to(BF), (rnd(g, P, K).abs() + 0.5).to(BF)
    dy[5, 3], dy[4000, 9], dy[70, 17] = math.inf, -math.inf, math.nan
    dy[100, 33], dy[101, 33] = math.inf, -math.inf
    W = rnd(g, N, K).to(BF)
    dW, db = torch.empty(N, K, device=DEV), torch.empty(N, device=DEV)
    o.linear_bwd(dy, x, K, W, None, 0, dW, db, need_dx=False)
    want = dy.double().sum(0)
    ok = want.isfinite()
    assert torch.equal(db.isfinite(), ok) and rel(db[ok], want[ok]) < 1e-5
    assert torch.equal(db[~ok].nan_to_num(7.0), want[~ok].float().nan_to_num(7.0))
    assert torch.equal(dW.isfinite().all(1), ok) and torch.equal(dW.isfinite().any(1), ok)


# ---- surfel attributes --------------------------------------------------------------

# a lattice, where many neighbours tie at the k_n-th distance (the smaller index is
# the nearer), coincident points, and counts just above each list length; against
# a brute-force search by (FP32 squared distance, index) with FP64 sums
@pytest.mark.parametrize("k_r,k_n", [(8, 9), (8, 12), (11, 16), (15, 17), (23, 24), (31, 32)])
@pytest.mark.parametrize("kind", ["lattice", "coincident", "few"])
def test_point_attributes_ties(kind, k_r, k_n):
    from paper_2408_15583_gb300 import api
    g = gen(k_r + k_n)
    if kind == "lattice":
        ax = torch.arange(9, device=DEV, dtype=torch.float32)
        pos = torch.cartesian_prod(ax, ax, ax[:2] * 0.75)
        pos = pos[torch.randperm(len(pos), generator=g, device=DEV)]
    elif kind == "coincident":
        pos = torch.rand(60, 3, generator=g, device=DEV).repeat(40, 1)
    else:
        pos = torch.rand(max(k_r + 1, k_n) + 1, 3, generator=g, device=DEV)
    pos = pos.contiguous()
    n = len(pos)
    rad, nrm = api.point_attributes(pos, k_r, k_n)
    api.stream_check()
    e = (pos[:, None] - pos[None]) ** 2
    d2 = (e[..., 0] + e[..., 1]) + e[..., 2]                 # the kernel's order
    key = d2.view(torch.int32).long() << 32 | torch.arange(n, device=DEV)[None]
    key = key.sort(1).values
    idx, d = key & 0xffffffff, (key >> 32).int().view(torch.float32).double()
    assert torch.equal(rad, (d[:, 1:k_r + 1].sqrt().sum(1) / k_r).float())
    nb = pos[idx[:, :k_n]].double()
    nb = nb - nb.mean(1, keepdim=True)
    val, vec = torch.linalg.eigh((nb.transpose(1, 2) @ nb).cpu())
    clear = (val[:, 1] - val[:, 0] > 1e-3 * val[:, 2]) & (val[:, 2] > 0)   # a defined normal
    dot = (vec[:, :, 0] * nrm.cpu().double()).sum(1).abs()[clear]
    # FP32 rounding of a unit vector: 1 - |dot| <= (2^-24 sqrt(3))^2 / 2 + FP64 noise
    # amplified by the gap bound (1e-16 / 1e-3)
    assert bool((dot > 1 - 1e-7).all())


# ---- pooling, sub-pixel shuffle, one-output heads -----------------------------------

@pytest.mark.parametrize("B,H,W,C", [(1, 2, 2, 8), (2, 6, 10, 40), (3, 34, 18, 64)])
def test_pool_and_shuffle(B, H, W, C):
    o, g = ops(), gen(B + H + W + C)
    x = rnd(g, B, H, W, C).to(BF)
    x[:, ::3] = x[:, ::3].round()                     # ties: the first of the four wins
    y = torch.empty(B, H // 2, W // 2, C, dtype=BF, device=DEV)
    arg = torch.empty(y.shape, dtype=torch.uint8, device=DEV)
    o.maxpool(x, B, H, W, C, y, arg)
    four = x.view(B, H // 2, 2, W // 2, 2, C).permute(0, 1, 3, 2, 4, 5).reshape(*y.shape[:3], 4, C)
    best = four.float().max(3).values
    assert torch.equal(y.float(), best)
    first = (four.float() == best[..., None, :]).float().argmax(3)
    assert torch.equal(arg.long(), first)
    dy, dx = rnd(g, *y.shape).to(BF), torch.empty_like(x)
    o.maxpool(dy, B, H, W, C, dx, arg, backward=True)
    want = torch.zeros_like(four).scatter_(3, first[..., None, :], dy[..., None, :])
    assert torch.equal(dx.view(B, H // 2, 2, W // 2, 2, C).permute(0, 1, 3, 2, 4, 5).reshape(four.shape),
                       want)
    # [B, H, W, 4 C] <-> channels 8 .. 8 + C of a [B, 2 H, 2 W, C + 24] image
    small = rnd(g, B, H, W, 4 * C).to(BF)
    big = torch.full((B, 2 * H, 2 * W, C + 24), 7.0, dtype=BF, device=DEV)
    o.shuffle(small, B, H, W, C, big, C + 24, 8)
    ref = torch.nn.functional.pixel_shuffle(small.permute(0, 3, 1, 2).float(), 2).permute(0, 2, 3, 1)
    assert torch.equal(big[..., 8:8 + C].float(), ref)
    assert bool((big[..., :8] == 7.0).all()) and bool((big[..., 8 + C:] == 7.0).all())
    back = torch.empty_like(small)
    o.shuffle(big, B, H, W, C, back, C + 24, 8, backward=True)
    assert torch.equal(back, small)


# layers of one to four outputs; FP32 sums over P products err below 1e-5, and the
# data gradient of a one-output layer is one product, rounded once to BF16
@pytest.mark.parametrize("N", [1, 2, 3, 4])
@pytest.mark.parametrize("P,K", [(1, 8), (63, 32), (100_001, 32), (5000, 256), (777, 40)])
def test_thin_layer_gradients(P, K, N):
    o, g = ops(), gen(P + K + N)
    dy, x, W = rnd(g, P, N).to(BF), rnd(g, P, K).to(BF), rnd(g, N, K).to(BF)
    dW, db = torch.empty(N, K, device=DEV), torch.empty(N, device=DEV)
    dx = torch.empty(P, K, dtype=BF, device=DEV)
    o.linear_bwd(dy, x, K, W, dx, K, dW, db)
    assert rel(dW, dy.double().T @ x.double()) < 1e-5 and rel(db, dy.double().sum(0)) < 1e-5
    if N == 1:
        assert torch.equal(dx, (dy.float() * W.float()).to(BF))
    else:
        assert rel(dx, dy.double() @ W.double()) < BF_TOL


# ---- 3x3 convolution ----------------------------------------------------------------

# channel counts gathered by the loads (multiples of 64) and not; images narrower
# than a tile of pixels, rows that end inside one, several images to a tile, and
# enough pixels for the unsplit kernel (128 outputs from 65536 pixels on)
@pytest.mark.parametrize("B,H,W,Cin,Cout", [(1, 1, 1, 64, 128), (3, 5, 7, 64, 72), (2, 8, 8, 40, 96),
                                            (5, 130, 101, 64, 128), (40, 41, 43, 128, 256)])
def test_conv3(B, H, W, Cin, Cout):
    from paper_2408_15583_gb300 import api
    o, g = ops(), gen(B + H + W + Cin)
    x = rnd(g, B, H, W, Cin).to(BF)
    w = (rnd(g, Cout, 3, 3, Cin) / math.sqrt(9 * Cin)).to(BF)
    b, dy = rnd(g, Cout), rnd(g, B * H * W, Cout).to(BF)
    y = torch.empty(B * H * W, Cout, dtype=BF, device=DEV)
    dW, db = torch.empty(Cout, 9 * Cin, device=DEV), torch.empty(Cout, device=DEV)
    o.conv3(x, w, b, B, H, W, Cin, Cout, y)
    o.conv3_wgrad(dy, x, B, H, W, Cin, Cout, dW, db)
    api.stream_check()
    xp = torch.nn.functional.pad(x.double(), (0, 0, 1, 1, 1, 1))
    col = torch.cat([xp[:, i:i + H, j:j + W] for i in range(3) for j in range(3)], -1).view(-1, 9 * Cin)
    assert rel(y, col @ w.double().view(Cout, -1).T + b.double()) < BF_TOL
    assert rel(dW, dy.double().T @ col) < 1e-5 and rel(db, dy.double().sum(0)) < 1e-5


@pytest.mark.parametrize("M,N,K", [(70000, 1, 64), (66000, 3, 64), (40963, 8, 72), (129, 2, 8)])
def test_narrow_fp32_output(M, N, K):
    from paper_2408_15583_gb300 import api
    o, g = ops(), gen(M + N)
    a, w, b = rnd(g, M, K).to(BF), rnd(g, N, K).to(BF), rnd(g, N)
    y = torch.full((M + 1, N), 7.0, device=DEV)
    o.gemm(M, N, K, a, K, 1, w, 1, K, y, N, bias=b)
    api.stream_check()
    ref = a.double() @ w.double().T + b.double()
    assert float((y[:M].double() - ref).abs().max()) < 2e-5 * K ** 0.5 and bool((y[M] == 7.0).all())


# ---- surfel attributes ----------------------------------------------------------------

# clouds inside and outside the range of the pair arithmetic, and shapes whose two
# smallest axes are close (the full solution) or not.  The normal is rounded to
# FP32, an angle of at most 1e-7 from the axis, and its own error adds less than as
# much again, so n'An exceeds the smallest eigenvalue by at most (2e-7)^2 of the
# largest; the radius is one rounding away, 2^-24.
@pytest.mark.parametrize("scale", [1e-12, 1e-7, 1.0, 1e9, 1e16])
@pytest.mark.parametrize("shape", [(1.0, 0.7, 0.05), (1.0, 0.02, 0.01), (1.0, 0.9, 0.8)])
def test_point_attributes_scales(scale, shape):
    import numpy as np
    from paper_2408_15583_gb300 import api
    rng, n, k_r, k_n = np.random.default_rng(7), 600, 8, 16
    pos = (rng.standard_normal((n, 3)) * np.array(shape) * scale + 3.0 * scale).astype(np.float32)
    rad, nrm = api.point_attributes(torch.tensor(pos, device=DEV), k_r, k_n, None, radius=True,
                                    normal=True)
    api.stream_check()
    rad, nrm = rad.double().cpu().numpy(), nrm.double().cpu().numpy()
    d = pos[:, None] - pos[None]
    d2 = (d[..., 0] * d[..., 0] + d[..., 1] * d[..., 1]) + d[..., 2] * d[..., 2]
    order = np.argsort(d2, axis=1, kind="stable")
    for i in range(n):
        r = np.sqrt(d2[i, order[i, 1:k_r + 1]].astype(np.float64)).mean()
        x = pos[order[i, :k_n]].astype(np.float64) - pos[i].astype(np.float64)
        x = (x - x.mean(0)) / scale
        A = x.T @ x
        lam = np.linalg.eigvalsh(A)
        assert abs(rad[i] - r) <= 1.01 * 2.0 ** -24 * r
        assert nrm[i] @ A @ nrm[i] / (nrm[i] @ nrm[i]) - lam[0] < 4.1e-14 * lam[2]


# one input channel: tiles of 16 pixels that end inside a row, an image or a warp's
# share; the forward products are those of the general contraction, bit for bit
@pytest.mark.parametrize("B,H,W,Cout", [(1, 1, 1, 32), (2, 3, 5, 64), (3, 17, 19, 32), (1, 260, 517, 32),
                                        (2, 9, 16, 8), (1, 40, 33, 128), (1, 12, 11, 40)])
def test_conv3_one_channel(B, H, W, Cout):
    from paper_2408_15583_gb300 import api
    o, g, P = ops(), gen(B + H + W + Cout), B * H * W
    x, b, dy = rnd(g, B, H, W, 1).to(BF), rnd(g, Cout), rnd(g, P, Cout).to(BF)
    w = (rnd(g, Cout, 9) / 3).to(BF)
    y, z, col = (torch.empty(P, n, dtype=BF, device=DEV) for n in (Cout, Cout, 9))
    dW, db = torch.empty(Cout, 9, device=DEV), torch.empty(Cout, device=DEV)
    o.conv3(x, w, b, B, H, W, 1, Cout, y)
    o.conv3_wgrad(dy, x, B, H, W, 1, Cout, dW, db)
    o.im2col(x, B, H, W, 1, col)
    o.gemm(P, Cout, 9, col, 9, 1, w, 1, 9, z, Cout, bias=b)
    api.stream_check()
    xp = torch.nn.functional.pad(x.double(), (0, 0, 1, 1, 1, 1))
    ref = torch.cat([xp[:, i:i + H, j:j + W] for i in range(3) for j in range(3)], -1).view(-1, 9)
    assert torch.equal(col.double(), ref) and torch.equal(y, z)
    assert rel(dW, dy.double().T @ ref) < 1e-5 and rel(db, dy.double().sum(0)) < 1e-5


# rows off 16-byte boundaries: the same bits
@pytest.mark.parametrize("Cout", [8, 32, 64, 128, 40])
def test_conv3_one_channel_unaligned(Cout):
    from paper_2408_15583_gb300 import api
    o, g, (B, H, W) = ops(), gen(Cout), (2, 21, 19)
    P = B * H * W
    x, b, dy = rnd(g, P).to(BF), rnd(g, Cout), rnd(g, P, Cout).to(BF)
    w = (rnd(g, Cout, 9) / 3).to(BF)

    def off(t):
        return torch.empty(t.numel() + 1, dtype=t.dtype, device=DEV)[1:].view(t.shape).copy_(t)

    res = []
    for f in (lambda t: t, off):
        y = f(torch.full((P, Cout), 7.0, dtype=BF, device=DEV))
        dW, db = torch.empty(Cout, 9, device=DEV), torch.empty(Cout, device=DEV)
        o.conv3(f(x), f(w), b, B, H, W, 1, Cout, y)
        o.conv3_wgrad(f(dy), f(x), B, H, W, 1, Cout, dW, db)
        api.stream_check()
        res.append((y, dW, db))
    assert torch.equal(res[0][0], res[1][0])
    assert rel(res[1][1], res[0][1]) < 1e-5 and rel(res[1][2], res[0][2]) < 1e-5
    if Cout != 40:
        assert torch.equal(res[0][1], res[1][1]) and torch.equal(res[0][2], res[1][2])


# two to eight splits and more, with and without a residual, whole rows of eight and not
@pytest.mark.parametrize("M,N,K", [(16384, 256, 1024), (1000, 64, 2304), (640, 136, 1100), (257, 36, 600)])
def test_split_contraction(M, N, K):
    from paper_2408_15583_gb300 import api
    o, g = ops(), gen(M + N)
    a, w = rnd(g, M, K).to(BF), (rnd(g, N, K) / math.sqrt(K)).to(BF)
    b, r = rnd(g, N), rnd(g, M, N).to(BF)
    y, y32 = torch.empty(M, N, dtype=BF, device=DEV), torch.empty(M, N, device=DEV)
    o.gemm(M, N, K, a, K, 1, w, 1, K, y, N, bias=b, R=r, ldr=N)
    o.gemm(M, N, K, a, K, 1, w, 1, K, y32, N)
    api.stream_check()
    ref = a.double() @ w.double().T
    assert rel(y32, ref) < 1e-5 and rel(y, ref + b.double() + r.double()) < BF_TOL


# ---- the network's parameter views ---------------------------------------------

# the layer calls' views belong to the buffers: a network whose buffers were
# replaced computes with the new ones, and so does one updated in place
@pytest.mark.parametrize("how", ["replaced", "in place"])
def test_parameter_views_follow_their_buffers(how):
    import scenes
    from paper_2408_15583_gb300.learned import UNet
    widths, blocks, H = (8, 8), (1, 1), 16
    a, b = (UNet(scenes.unet_init(seed, widths, blocks), widths, blocks, DEV) for seed in (1, 2))
    x = rnd(gen(3), H * H).to(BF)

    def step(net):
        outs, tape = net.forward(x, 1, H, H)
        net.backward(tape, {k: torch.ones_like(v) for k, v in outs.items()})
        return outs, net.grad.clone()

    before, _ = step(a)
    want, want_grad = step(b)
    for name in ("master", "mirror", "grad"):
        if how == "replaced":
            setattr(a, name, getattr(b, name).clone())
        else:
            getattr(a, name).copy_(getattr(b, name))
    got, got_grad = step(a)
    assert not torch.equal(before["depth"], want["depth"])
    for k in want:
        assert torch.equal(got[k], want[k])
    assert torch.equal(got_grad, want_grad)


# the gradients are those of the forward pass, whatever the caller did to its input
# in between
@pytest.mark.parametrize("widths,H", [((32, 64), 16), ((8,), 5)])
def test_gradients_after_the_input_was_overwritten(widths, H):
    import scenes
    from paper_2408_15583_gb300.learned import UNet
    blocks = (1,) * len(widths)
    net = UNet(scenes.unet_init(4, widths, blocks), widths, blocks, DEV)
    x = rnd(gen(5), H * H).to(BF)

    def step(overwrite):
        mine = x.clone()
        outs, tape = net.forward(mine, 1, H, H)
        if overwrite:
            mine.fill_(3.0)
        net.backward(tape, {k: torch.ones_like(v) for k, v in outs.items()})
        return net.grad.clone()

    assert torch.equal(step(False), step(True))


# a captured pass goes on writing the workspace it was captured with: a larger eager
# pass, which takes a larger one, leaves that memory to the graph
def test_captured_pass_keeps_its_workspace():
    import gc
    import scenes
    from paper_2408_15583_gb300.learned import GraphedUNet, UNet
    widths, blocks, H = (8, 16), (1, 1), 32
    net = UNet(scenes.unet_init(6, widths, blocks), widths, blocks, DEV)
    g = gen(7)
    x, big = rnd(g, H * H).to(BF), rnd(g, 16 * H * H).to(BF)
    graphed = GraphedUNet(net, 1, H, H)
    want = {k: v.clone() for k, v in graphed.forward(x).items()}
    at, size = net.ops._ws.data_ptr(), net.ops._ws.numel()
    net.forward(big, 16, H, H)
    assert net.ops._ws.data_ptr() != at
    gc.collect()
    others = [torch.full((size,), 7, dtype=torch.uint8, device=DEV) for _ in range(8)]
    got = graphed.forward(x)
    assert all(torch.equal(got[k], want[k]) for k in want)
    assert all(bool((t == 7).all()) for t in others)
    assert all(t.data_ptr() >= at + size or t.data_ptr() + size <= at for t in others)


# ---- Canny hysteresis over its tiles --------------------------------------------

# a weak depth step along a serpentine corridor, strong at its start only, on
# screens around the 64-pixel tiles: the edge follows the corridor through several
# tiles and passes, and the splats equal the oracle's bit for bit
@pytest.mark.parametrize("n", [8, 63, 64, 65, 129, 200])
def test_canny_edge_followed_over_tiles(n):
    import numpy as np
    import oracle
    from paper_2408_15583_gb300 import api
    from paper_2408_15583_gb300._lib import PeParams
    frame = ([0.0, 0.0, 5.0], [1.0, 0.0, 0.0], [0.0, 1.0, 0.0], [0.0, 0.0, -1.0])
    view = oracle.View(*(np.array(a) for a in frame), pitch=0.125, W=n, H=n)
    lane = np.zeros((n, n), bool)
    for k, r in enumerate(range(3, n - 6, 14)):
        lane[r:r + 6, 4:n - 4] = True
        lane[r:r + 20, (n - 10 if k % 2 == 0 else 4):][:, :6] = True
    lane[n - 3:] = False
    start = lane & (np.arange(n)[:, None] < 9) & (np.arange(n)[None] < 12)
    nrm = np.tile([0.0, 0.0, 1.0], (n * n, 1))

    def splats(depth):
        g = oracle.Gfb(depth=depth.ravel(), idx=np.zeros(n * n, np.int64), nrm=nrm, view=view, pix=None)
        fp = oracle.FuseParams(tau=3.0, bmin=np.array([-16.0, -16.0, -16.0]), inv_vox=8.0, G=256,
                               edge_mode=1)
        want = oracle.aggregate([g], fp, "fp32")
        nd = torch.from_numpy(np.concatenate([nrm, depth.reshape(-1, 1)], 1).astype(np.float32)).to(DEV)
        prm = PeParams(eps=0.125, overlap_r=0.125, edge_tau=3.0, fuse_grid=256,
                       bbox_min=(-16.0, -16.0, -16.0), inv_voxel=8.0, edge_mode=1)
        geom = api.aggregate_views([api.view_from_struct(*frame, 0.125, n, n)], nd,
                                   torch.ones(n * n, dtype=torch.uint8, device=DEV), prm)
        cr, _ = geom.planes()
        cr = cr.cpu().numpy()
        ids = np.flatnonzero(cr[:, 3] > 0)
        assert np.array_equal(ids, want.id)
        assert np.array_equal(cr[ids, :3].astype(np.float64), want.c)
        return ids

    weak = 5.0 + 0.875 * lane
    alone = splats(weak)
    followed = splats(np.where(start, 7.0, weak))
    if n >= 63:     # far more pixels become edges than the strong start's own rim
        assert len(alone) - len(followed) > 4 * n
