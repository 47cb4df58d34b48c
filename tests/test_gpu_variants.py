"""Kernel variants at the sizes where they can go wrong: edges of tiles and
chunks, remainders, operands off their fast path's alignment."""
import numpy as np
import pytest
import torch

from paper_2206_05085_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    from paper_2206_05085_gb300 import build
    build.build()
    from paper_2206_05085_gb300 import _lib
    return _lib


def _select_ref(q, off, n_draw):
    """The header's rule, one candidate at a time in FP32."""
    sel = np.full((len(off) - 1, n_draw), -1, np.int32)
    cnt = np.zeros(len(off) - 1, np.int32)
    u = ((np.arange(n_draw, dtype=np.float32) + np.float32(0.5)) / np.float32(n_draw)).astype(np.float32)
    for r in range(len(off) - 1):
        x = q[off[r]:off[r + 1]]
        if len(x) == 0:
            continue
        j, cdf, out = 0, x[0], []
        for k in range(n_draw):
            while j < len(x) - 1 and not (u[k] < cdf):
                j += 1
                cdf = np.float32(cdf + x[j])
            if not out or out[-1] != j:
                out.append(j)
        sel[r, :len(out)] = out
        cnt[r] = len(out)
    return sel, cnt


@pytest.mark.parametrize("n_draw", [1, 7, 64, 130])
def test_select_against_sequential_rule(L, n_draw):
    rng = np.random.default_rng(3)
    lens = [0, 1, 2, 3, 31, 32, 33, 127, 128, 129, 255, 256, 257, 0, 512, 5, 300]
    rows = []
    for i, n in enumerate(lens):
        x = rng.random(n).astype(np.float32) ** 4
        if n:
            x /= np.float32(max(x.sum(), 1e-6))
        if n > 4 and i % 4 == 0:
            x[n // 2] = np.nan            # the CDF is NaN from here: nothing exceeds it
        if n > 4 and i % 4 == 1:
            x[1::3] *= -1                 # a CDF that falls again
        if n > 4 and i % 4 == 2:
            x[n // 3] = np.inf
        rows.append(x)
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    q = np.concatenate(rows)
    with np.errstate(invalid="ignore"):
        ref_sel, ref_n = _select_ref(q, off, n_draw)
    R = len(lens)
    sel = torch.full((R * n_draw,), 7, dtype=torch.int32, device="cuda")
    n_sel = torch.full((R,), 7, dtype=torch.int32, device="cuda")
    L.proposal_select(torch.from_numpy(q).cuda(), torch.from_numpy(off).cuda(), R, n_draw, sel, n_sel)
    assert np.array_equal(n_sel.cpu().numpy(), ref_n)
    assert np.array_equal(sel.cpu().numpy().reshape(R, n_draw), ref_sel)


@pytest.mark.parametrize("precision", ["f32tc", "bf16"])
@pytest.mark.parametrize("n", [1, 127, 128, 129, 152 * 128 + 1])
def test_rgbnet_parameters_off_alignment(L, precision, n):
    """Parameters that start 4 bytes past a 16-byte boundary take the scalar
    weight loads: the same values, so the same bits."""
    P = {"f32tc": L.F32_TC, "bf16": L.BF16}[precision]
    g = torch.Generator(device="cuda").manual_seed(n)
    k0 = torch.randn(n, 12, generator=g, device="cuda") * 0.3
    d = torch.nn.functional.normalize(torch.randn(n // 7 + 1, 3, generator=g, device="cuda"), dim=1)
    ray = (torch.arange(n, device="cuda") // 7).int()
    up = torch.randn(n, 3, generator=g, device="cuda") * 1e-3
    p = torch.from_numpy(synth.mlp_params(seed=1)).cuda()
    shifted = torch.empty(p.numel() + 1, device="cuda")[1:]
    shifted.copy_(p)
    assert shifted.data_ptr() % 16 == 4
    got = []
    for params in (p, shifted):
        rgb = torch.empty(n, 3, device="cuda")
        act = torch.empty(L.rgbnet_act_bytes(n, P), dtype=torch.uint8, device="cuda")
        g_p, g_k0 = torch.zeros_like(p), torch.empty_like(k0)
        L.rgbnet_fwd(k0, d, ray, None, n, None, params, P, rgb, act)
        L.rgbnet_bwd(up, None, None, k0, d, ray, None, n, None, params, P, g_p, g_k0, act, rgb)
        got.append((rgb, g_p, g_k0))
    for a, b in zip(*got):
        assert torch.equal(a, b)


@pytest.mark.parametrize("n", [1, 129, 152 * 128, 152 * 128 + 1, 305 * 128 + 77])
def test_proposal_bwd_tile_counts(L, n):
    """One tile, one per CTA, an odd number per CTA (the two groups of
    epilogue warps get unequal shares), against torch in 64 bits on the stored
    BF16 parameters.  A sample whose ReLU input lies within the operands' reach
    of 0 may switch the unit: its share of the gradient is allowed as slack."""
    g = torch.Generator(device="cuda").manual_seed(n)
    xyz = torch.rand(n, 3, generator=g, device="cuda") * 2 - 1
    up = torch.randn(n, generator=g, device="cuda")
    p = torch.from_numpy(synth.proposal_params(2)).cuda()
    g_p = torch.zeros_like(p)
    L.proposal_bwd(up, xyz, None, n, None, p, g_p)
    assert L.device_status() == 0
    q = p.to(torch.bfloat16).double().requires_grad_()
    W1, b1, W2, b2, W3 = q[:2496].view(64, 39), q[2496:2560], q[2560:6656].view(64, 64), q[6656:6720], q[6720:6784]
    x = xyz.double()
    arg = (x[:, :, None] * 2.0 ** torch.arange(6, device="cuda", dtype=torch.float64)).flatten(1)
    z1 = torch.cat([x, arg.sin(), arg.cos()], 1) @ W1.T + b1
    z2 = torch.relu(z1) @ W2.T + b2
    z = torch.relu(z2) @ W3 + q[6784]
    (ref,) = torch.autograd.grad(z, q, up.double(), retain_graph=True)
    close = torch.minimum(z1.abs().amin(1), z2.abs().amin(1)) < 2e-5
    slack = torch.zeros_like(ref)
    for s in close.nonzero()[:, 0].tolist():
        (gs,) = torch.autograd.grad(z[s], q, up[s].double(), retain_graph=True)
        slack += 2 * gs.abs()
    tol = 2e-5 * ref.abs().max()   # two BF16 terms: 2^-16 of each factor
    assert bool(((g_p.double() - ref).abs() <= tol + slack).all())


@pytest.mark.parametrize("n_flat", [3, 4099, 22019])
@pytest.mark.parametrize("density", [0.0, 0.03, 0.5, 1.0])
def test_adam_list_against_single_arrays(L, n_flat, density):
    """The list kernel (flagged bricks of two grids and a flat vector with a
    cut last group and a short last block) against the call per array: the same
    arithmetic, so the same bits; unlisted bricks untouched, flags cleared."""
    nb, dev = 300, "cuda"
    g = torch.Generator(device=dev).manual_seed(n_flat)
    flags = (torch.rand(nb, generator=g, device=dev) < 0.4).to(torch.uint8)
    lst = torch.empty(nb, dtype=torch.int32, device=dev)
    cnt = torch.zeros(1, dtype=torch.int32, device=dev)
    L.touched_compact(flags, nb, lst, cnt)

    def state(n, dens):
        r = [torch.randn(n, generator=g, device=dev) for _ in range(4)]
        r[3] = r[3].abs()
        r[1] = r[1] * (torch.rand(n, generator=g, device=dev) < dens)
        return r   # p, g, m, v
    sets = [state(nb * 512, density), state(nb * 512 * 12, density), state(n_flat, 1.0)]
    sh = torch.zeros(nb * 512 * 12, dtype=torch.bfloat16, device=dev)
    ref = [[x.clone() for x in s] for s in sets]
    ref_sh, f = sh.clone(), [flags.clone() for _ in range(4)]
    step = torch.zeros(2, dtype=torch.int64, device=dev)
    step[0] = 4
    L.adam_step_multi_dev(
        [(s[0], sh if i == 1 else None, *s[1:], s[0].numel(), f[i] if i < 2 else None, 512 * (1, 12, 0)[i], 0.1,
          *((lst, cnt) if i < 2 else ())) for i, s in enumerate(sets)], 0.9, 0.99, 1e-15, step, True)
    for i, s in enumerate(ref):
        L.adam_step(s[0], ref_sh if i == 1 else None, *s[1:], s[0].numel(), f[2 + i] if i < 2 else None,
                    512 * (1, 12, 0)[i], 0.1, 0.9, 0.99, 1e-15, 5, True)
    assert int(step[0]) == 5
    for a, b in zip(sets, ref):
        for x, y in zip(a, b):
            assert torch.equal(x, y)
    assert torch.equal(sh, ref_sh)
    assert int(f[0].sum()) == 0 and int(f[1].sum()) == 0


@pytest.mark.parametrize("listed", [1, 557, 561, 562, 565, 2000, 5000])   # both sides of one piece a warp; many pieces
@pytest.mark.parametrize("density", [0.03, 0.5, 1.0])
@pytest.mark.parametrize("zero_grad", [True, False])
def test_adam_list_lengths(L, listed, density, zero_grad):
    """The list kernel at lengths of either of its loops, with whole bricks and
    single groups of zero gradients, against the call per array: the same bits,
    flags cleared (or, without zero_grad, gradients and flags kept)."""
    nb, dev = 5003, "cuda"
    g = torch.Generator(device=dev).manual_seed(listed)
    flags = torch.zeros(nb, dtype=torch.uint8, device=dev)
    flags[torch.randperm(nb, generator=g, device=dev)[:listed]] = 1
    lst, cnt = torch.empty(nb, dtype=torch.int32, device=dev), torch.zeros(1, dtype=torch.int32, device=dev)
    L.touched_compact(flags, nb, lst, cnt)

    def state(C):
        p, m = (torch.randn(nb * 512 * C, generator=g, device=dev) for _ in range(2))
        grad = torch.randn(nb * 512 * C, generator=g, device=dev)
        keep = (torch.rand(nb * 128 * C, generator=g, device=dev) < density).repeat_interleave(4)
        keep &= (torch.rand(nb, generator=g, device=dev) < 0.9).repeat_interleave(512 * C)
        return [p, grad * keep, m, m.abs()]
    sets = [state(1), state(12)]
    ref = [[x.clone() for x in s] for s in sets]
    f = [flags.clone() for _ in range(4)]
    L.adam_step_multi([(s[0], None, *s[1:], s[0].numel(), f[i], 512 * (1, 12)[i], 0.1, lst, cnt)
                       for i, s in enumerate(sets)], 0.9, 0.99, 1e-15, 3, zero_grad)
    for i, s in enumerate(ref):
        L.adam_step(s[0], None, *s[1:], s[0].numel(), f[2 + i], 512 * (1, 12)[i], 0.1, 0.9, 0.99, 1e-15, 3, zero_grad)
    for a, b in zip(sets, ref):
        for x, y in zip(a, b):
            assert torch.equal(x, y)
    assert all(torch.equal(x, torch.zeros_like(flags) if zero_grad else flags) for x in f)


@pytest.mark.parametrize("G", [(61, 47, 53), (8, 8, 8), (9, 16, 17)])
@pytest.mark.parametrize("bf16", [False, True])
def test_tv_pair_against_single_grids(L, G, bf16):
    """The paired sparse TV over the brick list against the call per grid: the
    same arithmetic, so the same bits (sides no multiple of the brick, empty
    and full bricks, entries zero in some channels)."""
    dev, nb = "cuda", L.grid_num_bricks(G)
    g = torch.Generator(device=dev).manual_seed(sum(G))
    flags = (torch.rand(nb, generator=g, device=dev) < 0.7).to(torch.uint8)
    flags[0] = 1
    lst = torch.empty(nb, dtype=torch.int32, device=dev)
    cnt = torch.zeros(1, dtype=torch.int32, device=dev)
    L.touched_compact(flags, nb, lst, cnt)
    dt = L.BF16 if bf16 else L.F32
    grids, ref = [], []
    for C, w in ((12, 1e-3), (1, 1e-2)):
        dense = torch.randn(G[2], G[1], G[0], C, generator=g, device=dev).to(torch.bfloat16 if bf16 else torch.float32)
        p = torch.empty(L.grid_bricked_elems(G, C), dtype=dense.dtype, device=dev)
        L.grid_pack(dense, p, G, C, dt)
        up = torch.randn(G[2], G[1], G[0], C, generator=g, device=dev)
        up = up * (torch.rand(G[2], G[1], G[0], 1, generator=g, device=dev) < 0.3)
        up = up * (torch.rand(up.shape, generator=g, device=dev) < 0.8)
        gg = torch.empty(L.grid_bricked_elems(G, C), device=dev)
        L.grid_pack(up, gg, G, C, L.F32)
        grids.append((p, dt, C, w, flags, gg))
        ref.append(gg.clone())
        L.tv_add_grad(p, dt, G, C, w, 0.5, False, flags, ref[-1])
    L.tv_add_grad_multi(grids, G, 0.5, False, lst, cnt)
    for (_, _, _, _, _, gg), r in zip(grids, ref):
        assert torch.equal(gg, r)


@pytest.mark.parametrize("n", [1, 127, 128, 129, 152 * 128 + 5])
@pytest.mark.parametrize("saved", [True, False])
def test_rgbnet_f32_tiles(L, n, saved):
    """The CUDA-core form at tile edges, with and without the stored
    activations, against torch in 64 bits.  FP32 sums of at most 128 terms: 1e-5
    of the largest value (a unit whose input lies within 1e-6 of 0 may switch;
    its samples are set aside, their share of the gradient allowed as slack)."""
    dev = "cuda"
    g = torch.Generator(device=dev).manual_seed(n)
    k0 = torch.randn(n, 12, generator=g, device=dev) * 0.3
    d = torch.nn.functional.normalize(torch.randn(n // 5 + 1, 3, generator=g, device=dev), dim=1)
    ray = (torch.arange(n, device=dev) // 5).int()
    up = torch.randn(n, 3, generator=g, device=dev)
    p = torch.from_numpy(synth.mlp_params(seed=4)).to(dev)
    rgb, act = torch.empty(n, 3, device=dev), torch.full((n, 256), -7.0, device=dev) if saved else None
    g_p, g_k0 = torch.zeros_like(p), torch.empty_like(k0)
    L.rgbnet_fwd(k0, d, ray, None, n, None, p, L.F32, rgb, act)
    L.rgbnet_bwd(up, None, None, k0, d, ray, None, n, None, p, L.F32, g_p, g_k0, act, rgb if saved else None)
    q = p.double().requires_grad_()
    x0 = k0.double().requires_grad_()
    at, W = 0, []
    for s in ((128, 39), (128,), (128, 128), (128,), (3, 128), (3,)):
        m = int(np.prod(s))
        W.append(q[at:at + m].view(s))
        at += m
    dd = d.double()[ray.long()]
    arg = (dd[:, :, None] * 2.0 ** torch.arange(4, device=dev, dtype=torch.float64)).flatten(1)
    z1 = torch.cat([x0, dd, arg.sin(), arg.cos()], 1) @ W[0].T + W[1]
    z2 = torch.relu(z1) @ W[2].T + W[3]
    y = torch.sigmoid(torch.relu(z2) @ W[4].T + W[5])
    r_p, r_k0 = torch.autograd.grad(y, (q, x0), up.double(), retain_graph=True)
    close = torch.minimum(z1.abs().amin(1), z2.abs().amin(1)) < 1e-6
    slack = torch.zeros_like(r_p)
    for s in close.nonzero()[:, 0].tolist():
        (gs,) = torch.autograd.grad(y[s], q, up[s].double(), retain_graph=True)
        slack += 2 * gs.abs()
    assert float((rgb.double() - y).abs().max()) <= 1e-5
    assert bool(((g_k0.double() - r_k0).abs().amax(1)[~close] <= 1e-5 * r_k0.abs().max()).all())
    assert bool(((g_p.double() - r_p).abs() <= 1e-5 * r_p.abs().max() + slack).all())
    if saved:
        assert float((act[:, :128].double() - torch.relu(z1)).abs().max()) <= 1e-5 * float(z1.abs().max())
        assert float((act[:, 128:].double() - torch.relu(z2)).abs().max()) <= 1e-5 * float(z2.abs().max())


@pytest.mark.parametrize("G", [(9, 10, 11), (64, 40, 33)])   # crowded (over half a sample per voxel) and not
@pytest.mark.parametrize("n", [1, 31, 33, 257, 4099])
@pytest.mark.parametrize("form", ["a", "b", "ab"])
def test_scatter_merge(L, G, n, form):
    """The merged adjoints (one channel, twelve, both) on runs of samples in one
    cell, an index list with a device count below the capacity, against a 64-bit
    scatter.  FP32 sums of at most n terms per voxel: 1e-5 of the largest entry."""
    dev = "cuda"
    g = torch.Generator(device=dev).manual_seed(n + G[0])
    base = torch.rand(n // 3 + 1, 3, generator=g, device=dev) * 2.2 - 1.1      # some outside the box
    xyz = (base.repeat_interleave(3, 0)[:n] + 0.01 * torch.rand(n, 3, generator=g, device=dev)).contiguous()
    ga = torch.randn(n, generator=g, device=dev)
    gb = torch.randn(n, 12, generator=g, device=dev)
    idx = torch.arange(n, device=dev, dtype=torch.int32).flip(0).contiguous()
    m = n - n // 5
    n_dev = torch.tensor([m], dtype=torch.int64, device=dev)
    gd = L.GridDesc.make(-1.0, 1.0, G)
    out = [torch.zeros(L.grid_bricked_elems(G, C), device=dev) for C in (1, 12)]
    flags = [torch.zeros(L.grid_num_bricks(G), dtype=torch.uint8, device=dev) for _ in range(2)]
    if form == "ab":
        L.sample_grid_bwd2(ga, 1, out[0], flags[0], gb, 12, out[1], flags[1], gd, xyz, idx, n, n_dev)
    elif form == "a":
        L.sample_grid_bwd(ga, gd, 1, xyz, idx, n, n_dev, out[0], flags[0])
    else:
        L.sample_grid_bwd(gb, gd, 12, xyz, idx, n, n_dev, out[1], flags[1])
    sel = idx[:m].long()
    dim = torch.tensor(G, device=dev)
    u = ((xyz[sel].double() + 1) * 0.5 * (dim - 1)).clamp(min=0)
    u = torch.minimum(u, (dim - 1).double())
    i = torch.minimum(u.floor().long(), dim - 2)
    f = u - i
    for C, up, got, fl in ((1, ga[:, None], out[0], flags[0]), (12, gb, out[1], flags[1])):
        ref = torch.zeros(G[2] * G[1] * G[0], C, dtype=torch.float64, device=dev)
        if {1: "a", 12: "b"}[C] in form:
            for k in range(8):
                o = torch.tensor([k & 1, (k >> 1) & 1, k >> 2], device=dev)
                w = torch.where(o.bool(), f, 1 - f).prod(1, keepdim=True)
                c = i + o
                ref.index_add_(0, (c[:, 2] * G[1] + c[:, 1]) * G[0] + c[:, 0], w * up[sel].double())
        dense = torch.empty(G[2], G[1], G[0], C, device=dev)
        L.grid_unpack(got, dense, G, C, L.F32)
        assert float((dense.view(-1, C).double() - ref).abs().max()) <= 1e-5 * max(float(ref.abs().max()), 1.0)
        hit = torch.zeros(G[2], G[1], G[0], dtype=torch.bool, device=dev)
        hit[(ref.abs().amax(1) > 0).view(G[2], G[1], G[0])] = True
        nb = [(x + 7) // 8 for x in G]
        full = torch.zeros(8 * nb[2], 8 * nb[1], 8 * nb[0], dtype=torch.bool, device=dev)
        full[:G[2], :G[1], :G[0]] = hit
        want = full.view(nb[2], 8, nb[1], 8, nb[0], 8).permute(0, 2, 4, 1, 3, 5).reshape(-1, 512).any(1)
        assert bool((fl.bool() | ~want).all())    # every brick with a contribution is flagged


@pytest.mark.parametrize("bad", [float("inf"), float("nan")])
@pytest.mark.parametrize("form", ["a", "b", "ab"])
def test_scatter_merge_nonfinite_rows(L, form, bad):
    """A row whose gradient is infinite or NaN reaches the eight voxels of its
    own cell and no others, wherever it stands in a warp's 32 samples and in a
    run of samples of one cell: the other voxels are the finite rows' 64-bit
    scatter (as in test_scatter_merge: 1e-5 of the largest entry)."""
    dev, G, n = "cuda", (40, 33, 35), 1003
    g = torch.Generator(device=dev).manual_seed(5)
    base = torch.rand(n, 3, generator=g, device=dev) * 1.9 - 0.95
    run = torch.randint(0, n, (n,), generator=g, device=dev).sort().values     # runs of one to several samples a cell
    xyz = (base[run] + 0.001 * torch.rand(n, 3, generator=g, device=dev)).contiguous()
    ga, gb = torch.randn(n, generator=g, device=dev), torch.randn(n, 12, generator=g, device=dev)
    rows = torch.arange(7, n, 37, device=dev)      # every position modulo 32
    fin_a, fin_b = ga.clone(), gb.clone()
    fin_a[rows], fin_b[rows] = 0.0, 0.0
    ga[rows], gb[rows] = bad, bad
    gd = L.GridDesc.make(-1.0, 1.0, G)
    out = [torch.zeros(L.grid_bricked_elems(G, C), device=dev) for C in (1, 12)]
    if form == "ab":
        L.sample_grid_bwd2(ga, 1, out[0], None, gb, 12, out[1], None, gd, xyz, None, n, None)
    elif form == "a":
        L.sample_grid_bwd(ga, gd, 1, xyz, None, n, None, out[0], None)
    else:
        L.sample_grid_bwd(gb, gd, 12, xyz, None, n, None, out[1], None)
    dim = torch.tensor(G, device=dev)
    u = (xyz.double() + 1) * 0.5 * (dim - 1)
    i = u.floor().long()
    f = u - i
    for C, up, got in ((1, fin_a[:, None], out[0]), (12, fin_b, out[1])):
        if {1: "a", 12: "b"}[C] not in form:
            continue
        ref = torch.zeros(G[2] * G[1] * G[0], C, dtype=torch.float64, device=dev)
        own = torch.zeros(G[2] * G[1] * G[0], dtype=torch.bool, device=dev)   # voxels of the bad rows' cells
        for k in range(8):
            o = torch.tensor([k & 1, (k >> 1) & 1, k >> 2], device=dev)
            w = torch.where(o.bool(), f, 1 - f).prod(1, keepdim=True)
            at = ((i + o)[:, 2] * G[1] + (i + o)[:, 1]) * G[0] + (i + o)[:, 0]
            ref.index_add_(0, at, w * up.double())
            own[at[rows]] = True
        dense = torch.empty(G[2], G[1], G[0], C, device=dev)
        L.grid_unpack(got, dense, G, C, L.F32)
        diff = (dense.view(-1, C).double() - ref).abs()[~own]
        assert bool((diff <= 1e-5 * float(ref.abs().max())).all())     # (NaN compares false)


@pytest.mark.parametrize("form", ["a", "b", "ab"])
def test_scatter_merge_second_trip(L, form):
    """More samples than the launch's warps take at once (2432 x 8 warps of 32):
    a warp's rows in shared memory are written again.  Sums of at most some
    hundred FP32 terms per voxel: 1e-5 of the largest entry; the flags are
    exactly the bricks of the samples' cells."""
    dev, n, G = "cuda", 650_001, (61, 70, 83)
    g = torch.Generator(device=dev).manual_seed(6)
    base = torch.rand(n // 2 + 1, 3, generator=g, device=dev) * 0.9 - 0.8     # a part of the grid
    xyz = (base.repeat_interleave(2, 0)[:n] + 0.004 * torch.rand(n, 3, generator=g, device=dev)).contiguous()
    ga, gb = torch.randn(n, generator=g, device=dev), torch.randn(n, 12, generator=g, device=dev)
    gd = L.GridDesc.make(-1.0, 1.0, G)
    out = [torch.zeros(L.grid_bricked_elems(G, C), device=dev) for C in (1, 12)]
    fl = [torch.zeros(L.grid_num_bricks(G), dtype=torch.uint8, device=dev) for _ in range(2)]
    if form == "ab":
        L.sample_grid_bwd2(ga, 1, out[0], fl[0], gb, 12, out[1], fl[1], gd, xyz, None, n, None)
    elif form == "a":
        L.sample_grid_bwd(ga, gd, 1, xyz, None, n, None, out[0], fl[0])
    else:
        L.sample_grid_bwd(gb, gd, 12, xyz, None, n, None, out[1], fl[1])
    dim = torch.tensor(G, device=dev)
    u = (xyz.double() + 1) * 0.5 * (dim - 1)
    i, nb = u.floor().long(), [(x + 7) // 8 for x in G]
    f = u - i
    want = torch.zeros(L.grid_num_bricks(G), dtype=torch.uint8, device=dev)
    ref = {C: torch.zeros(G[2] * G[1] * G[0], C, dtype=torch.float64, device=dev) for C in (1, 12)}
    for k in range(8):
        c = i + torch.tensor([k & 1, (k >> 1) & 1, k >> 2], device=dev)
        w = torch.where((c > i), f, 1 - f).prod(1, keepdim=True)
        want[((c[:, 2] >> 3) * nb[1] + (c[:, 1] >> 3)) * nb[0] + (c[:, 0] >> 3)] = 1
        for C, up in ((1, ga[:, None]), (12, gb)):
            ref[C].index_add_(0, (c[:, 2] * G[1] + c[:, 1]) * G[0] + c[:, 0], w * up.double())
    for C, got, flags, name in ((1, out[0], fl[0], "a"), (12, out[1], fl[1], "b")):
        if name not in form:
            continue
        dense = torch.empty(G[2], G[1], G[0], C, device=dev)
        L.grid_unpack(got, dense, G, C, L.F32)
        assert float((dense.view(-1, C).double() - ref[C]).abs().max()) <= 1e-5 * float(ref[C].abs().max())
        assert torch.equal(flags, want)


def test_tv_pair_second_trip(L):
    """Several 64-voxel units per warp: as test_tv_pair_against_single_grids."""
    test_tv_pair_against_single_grids(L, (160, 131, 150), False)


def test_select_second_trip(L):
    """More rays than the launch's warps take at once (2432 x 2 warps of four)."""
    rng = np.random.default_rng(9)
    R, n_draw = 20_011, 5
    lens = rng.integers(0, 9, R)
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    q = rng.random(int(off[-1])).astype(np.float32) * 0.3
    ref_sel, ref_n = _select_ref(q, off, n_draw)
    sel = torch.full((R * n_draw,), 7, dtype=torch.int32, device="cuda")
    n_sel = torch.full((R,), 7, dtype=torch.int32, device="cuda")
    L.proposal_select(torch.from_numpy(q).cuda(), torch.from_numpy(off).cuda(), R, n_draw, sel, n_sel)
    assert np.array_equal(n_sel.cpu().numpy(), ref_n)
    assert np.array_equal(sel.cpu().numpy().reshape(R, n_draw), ref_sel)


def _off_by(t, shift):
    """t's values in a view that starts `shift` elements past a 16-byte boundary."""
    v = torch.empty(t.numel() + shift, dtype=t.dtype, device=t.device)[shift:]
    v.copy_(t.reshape(-1))
    assert v.data_ptr() % 16 == shift * t.element_size()
    return v


@pytest.mark.parametrize("which", ["grid", "rows", "both"])
@pytest.mark.parametrize("bf16", [False, True])
def test_query12_off_alignment(L, bf16, which):
    """The 12-channel query and its adjoints (single and paired) on grids and
    rows that start one element past a 16-byte boundary: such buffers take the
    one-value-at-a-time kernels.  FP32 sums of 8 products (query) and of at most
    n terms (adjoint): 1e-6 and 1e-5 of the largest value."""
    dev, G, n = "cuda", (21, 18, 25), 2055
    g = torch.Generator(device=dev).manual_seed(8)
    xyz = (torch.rand(n, 3, generator=g, device=dev) * 2.2 - 1.1).contiguous()
    gd = L.GridDesc.make(-1.0, 1.0, G)
    dt, tdt = (L.BF16, torch.bfloat16) if bf16 else (L.F32, torch.float32)
    grid = torch.randn(L.grid_bricked_elems(G, 12), generator=g, device=dev).to(tdt)
    sg, sr = int(which != "rows"), int(which != "grid")
    want, got = torch.empty(n * 12, device=dev), _off_by(torch.zeros(n * 12, device=dev), sr)
    L.sample_grid_fwd(grid, dt, gd, 12, xyz, None, n, None, want)
    L.sample_grid_fwd(_off_by(grid, sg), dt, gd, 12, xyz, None, n, None, got)
    assert float((got - want).abs().max()) <= 1e-6 * float(want.abs().max())
    ga, gb = torch.randn(n, generator=g, device=dev), torch.randn(n * 12, generator=g, device=dev)
    ref = [torch.zeros(L.grid_bricked_elems(G, C), device=dev) for C in (1, 12)]
    fl = [torch.zeros(L.grid_num_bricks(G), dtype=torch.uint8, device=dev) for _ in range(6)]
    L.sample_grid_bwd2(ga, 1, ref[0], fl[0], gb, 12, ref[1], fl[1], gd, xyz, None, n, None)
    up = _off_by(gb, sr)
    one = _off_by(torch.zeros_like(ref[1]), sg)
    L.sample_grid_bwd(up, gd, 12, xyz, None, n, None, one, fl[2])
    pair = [torch.zeros_like(ref[0]), _off_by(torch.zeros_like(ref[1]), sg)]
    L.sample_grid_bwd2(ga, 1, pair[0], fl[3], up, 12, pair[1], fl[4], gd, xyz, None, n, None)
    for r, x in ((ref[1], one), (ref[0], pair[0]), (ref[1], pair[1])):
        assert float((x - r).abs().max()) <= 1e-5 * float(r.abs().max())
    for f in fl[1:5]:
        assert torch.equal(f, fl[0])


@pytest.mark.parametrize("which", ["grid", "gradient", "both"])
@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("dense", [False, True])
def test_tv_off_alignment(L, dense, bf16, which):
    """TV of grids and gradients that start one element past a 16-byte boundary
    (one channel at a time) against the aligned buffers: the same arithmetic per
    entry, so the same bits; single, and paired with a density grid over the
    brick list."""
    dev, G = "cuda", (19, 23, 10)
    nb = L.grid_num_bricks(G)
    g = torch.Generator(device=dev).manual_seed(2)
    dt, tdt = (L.BF16, torch.bfloat16) if bf16 else (L.F32, torch.float32)
    sp, sg = int(which != "gradient"), int(which != "grid")
    flags = (torch.rand(nb, generator=g, device=dev) < 0.7).to(torch.uint8)
    flags[0] = 1
    lst, cnt = torch.empty(nb, dtype=torch.int32, device=dev), torch.zeros(1, dtype=torch.int32, device=dev)
    L.touched_compact(flags, nb, lst, cnt)
    p = {C: torch.randn(nb * 512 * C, generator=g, device=dev).to(tdt) for C in (1, 4, 12)}
    up = {C: torch.randn(nb * 512 * C, generator=g, device=dev)
          * (torch.rand(nb * 512 * C, generator=g, device=dev) < 0.4) for C in (1, 4, 12)}
    for C in (4, 12):
        want, got = up[C].clone(), _off_by(up[C], sg)
        L.tv_add_grad(p[C], dt, G, C, 1e-3, 0.5, dense, flags.clone(), want)
        L.tv_add_grad(_off_by(p[C], sp), dt, G, C, 1e-3, 0.5, dense, flags.clone(), got)
        assert torch.equal(got, want) and not torch.equal(want, up[C])
    want = [up[1].clone(), up[12].clone()]
    got = [_off_by(up[1], sg), _off_by(up[12], sg)]
    for gr, off in ((want, 0), (got, 1)):
        L.tv_add_grad_multi([(_off_by(p[C], off * sp), dt, C, 1e-3, flags.clone(), x) for C, x in zip((1, 12), gr)],
                            G, 0.5, dense, None if dense else lst, None if dense else cnt)
    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])


@pytest.mark.parametrize("shift", [0, 1], ids=["aligned", "unaligned"])
@pytest.mark.parametrize("R", [1, 31, 1023, 1024, 1025, 8192, 8193, 152 * 1024 + 1, 400_001])
def test_count_scan_blocks(L, R, shift):
    """Live-sample list over per-ray counts whose scan is split over blocks:
    one to three passes a block, a last block of one ray, counts off 16-byte
    alignment."""
    rng = np.random.default_rng(R)
    cand = rng.integers(0, 6, R)
    live = np.minimum(rng.integers(0, 6, R), cand).astype(np.int32)
    off = np.concatenate([[0], np.cumsum(cand)]).astype(np.int64)
    seg = torch.from_numpy(np.concatenate([np.zeros(shift, np.int32), live])).cuda()[shift:]
    n = int(live.sum())
    idx = torch.full((max(n, 1),), -1, dtype=torch.int32, device="cuda")
    count = torch.zeros(1, dtype=torch.int64, device="cuda")
    ws = torch.empty(L.live_samples_workspace_size(R), dtype=torch.uint8, device="cuda")
    L.live_samples(torch.from_numpy(off).cuda(), seg, R, idx, count, ws)
    assert int(count) == n
    dst = np.concatenate([[0], np.cumsum(live)])[:-1]
    want = np.arange(n) + np.repeat(off[:-1] - dst, live)
    assert np.array_equal(idx.cpu().numpy()[:n], want)


@pytest.mark.parametrize("shift", [0, 1], ids=["aligned", "unaligned"])
@pytest.mark.parametrize("R", [7, 8, 9, 255, 256, 257, 4095, 4096, 4097])
def test_count_scan_small(L, R, shift):
    """The one-block scan: remainders of a thread's eight counts, a last thread
    of a warp, and both sides of its largest length."""
    test_count_scan_blocks(L, R, shift)


@pytest.mark.parametrize("steps", [1, 7, 8, 61, 130, 512])
@pytest.mark.parametrize("R", [1, 31, 33, 300])
def test_contracted_fill_groups(L, R, steps):
    """The contracted march's second pass from checkpoints (eight steps at a
    time, a warp writing four rays at once) against the march that writes as
    it goes: chunks shorter than a group, remainders, a ragged last block,
    sparse and full occupancy."""
    cfg = synth.CONFIGS["unbounded_320"]
    rp = synth.render_params(cfg)
    sd = L.SamplerDesc()
    sd.mode, sd.near, sd.max_steps = 1, rp.near, steps
    sd.contract_b, sd.p_inf, sd.step_c = rp.contract_b, steps % 2, rp.step_c * 4
    gd = L.GridDesc.make(cfg.bbox_min, cfg.bbox_max, [40] * 3)
    o, d = (torch.from_numpy(np.ascontiguousarray(v)).cuda() for v in synth.rays(cfg, seed=R, n_rays=R))
    n = R * steps
    for mask in (None, (torch.rand(40, 40, 40, generator=torch.Generator().manual_seed(1)) < 0.4)
                 .to(torch.uint8).cuda()):
        outs = []
        for _ in range(2):
            outs.append([torch.full((R + 1,), -1, dtype=torch.int64, device="cuda"),
                         torch.full((n, 3), -1.0, device="cuda"),
                         torch.full((n,), -1, dtype=torch.int32, device="cuda"),
                         torch.full((n,), -1, dtype=torch.int32, device="cuda"),
                         torch.full((n,), -1.0, device="cuda"), torch.full((n,), -1.0, device="cuda")])
        ws = torch.empty(L.sample_rays_workspace_size(R), dtype=torch.uint8, device="cuda")
        L.sample_rays(o, d, R, gd, sd, mask, n, *outs[0], ws)
        L.sample_rays_noalloc(o, d, R, gd, sd, mask, n, *outs[1])
        assert int(outs[0][0][-1]) > 0 or mask is not None
        for a, b in zip(*outs):
            assert torch.equal(a, b)
