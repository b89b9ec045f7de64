"""The hyperbatch's kernels at the sizes where they can go wrong -- edges of
tiles, remainders, the smallest and largest of a rule's range -- bit-exact
against the oracle, and the consumer layer within the oracle's bound."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
from agnes_inputs import synth
from paper_2601_01473_gb300 import AgnesError, Graph, lib
from test_gpu_parity import compare
from test_gpu_sage import _check_layer, _weights

pytestmark = pytest.mark.gpu


def _targets(N, H, B, seed):
    """H rows of B distinct ids (rows may share ids)."""
    gen = torch.Generator().manual_seed(seed)
    return torch.stack([torch.randperm(N, generator=gen)[:B] for _ in range(H)]).to(torch.int32)


def _graph(N, deg, dim, seed, block, dtype=torch.float16, bits=64, device="cuda:0"):
    off, ind = synth.rmat_csr(N, deg, 0.57, 0.19, 0.19, seed,
                              offsets_dtype=torch.int32 if bits == 32 else torch.int64)
    feats = synth.normal_features(N, dim, dtype, seed + 1)
    g = Graph(off.to(device), ind.to(device), feats.to(device), adj_block_bytes=block,
              feat_block_bytes=max(block, dim * feats.element_size()))
    return g, oracle.Graph(off.numpy(), ind.numpy(), feats.numpy()), off, ind, feats


@pytest.mark.parametrize("frontier", ["src", "sampled"])
@pytest.mark.parametrize("N,deg,H,B,fan", [
    (40, 6, 2, 3, [2, 2]),          # one tile, cells of a few entries
    (300, 30, 3, 4, [2, 3]),        # cells around the 4- and 8-entry networks
    (300, 30, 3, 20, [2, 3, 4]),    # around 32 frontier and 64 sampled entries
    (4096, 40, 2, 700, [4, 3]),     # one full tile, cells of thousands
    (4097, 20, 1, 900, [5, 2]),     # a second tile of one id
])
def test_cells_of_every_size(cuda_device, frontier, N, deg, H, B, fan):
    block = 1 << 20  # one block: the tiles are the 4096-id chunks
    g, og, *_ = _graph(N, deg, 16, N + deg, block)
    g.set_frontier(frontier)
    for seed in (1, 2):
        t = _targets(N, H, B, seed)
        g.prepare(t.to(cuda_device), fan, seed, 5)
        compare(g, og, t.numpy(), fan, seed, 5, block, block, frontier=frontier)
    g.close()


@pytest.mark.parametrize("H,B,block", [
    (1, 70_000, 1 << 16),   # 35 indptr tiles of one minibatch: two look-back windows
    (3, 2_047, 1 << 12),    # one row short of an indptr tile, many tiles of cells
    (5, 2_049, 1 << 12),    # one past it; 5 columns in the column scans
    (33, 300, 1 << 13),     # 33 columns: 64 wide
    (130, 40, 1 << 12),     # two column blocks
    (1, 1, 1 << 10), (1, 256, 1 << 12), (1, 257, 1 << 12), (16, 16, 1 << 12), (2, 129, 1 << 12),
])
def test_hyperbatch_shapes(cuda_device, H, B, block):
    N = 100_000
    g, og, *_ = _graph(N, 6, 16, 3, block, bits=32)
    t = _targets(N, H, B, H + B)
    for seed in (1, 2):
        g.prepare(t.to(cuda_device), [3], seed, 9)
        compare(g, og, t.numpy(), [3], seed, 9, block, block)
    g.close()


@pytest.mark.parametrize("H,first,B", [
    (5, 0, 64), (5, 0, 65),          # cells at the walk's limit and past it
    (2, 0, 255), (2, 100, 257), (1, 0, 513),
    (3, 4096, 4095), (2, 4096, 4096),  # all of a tile's ids but one, and all
    (2, 4000, 9000),                 # several large cells in a minibatch
    (70, 4090, 70),                  # cells of 6 and of 64
])
def test_targets_in_dense_cells(cuda_device, H, first, B):
    """Consecutive targets in random order, so that a (tile, minibatch) cell
    holds many; then one of them twice."""
    N, block = 20_000, 1 << 20  # one block: the tiles are the 4096-id chunks
    g, og, *_ = _graph(N, 6, 16, 5, block, bits=32)
    gen = torch.Generator().manual_seed(B)
    t = torch.stack([first + torch.randperm(B, generator=gen) for _ in range(H)]).to(torch.int32)
    bad = t.clone()
    bad[H - 1, B - 1] = bad[H - 1, 0]
    for targets in (t, bad, t):
        g.prepare(targets.to(cuda_device), [2], 4, 1)
        if targets is bad:
            with pytest.raises(AgnesError) as e:
                g.fetch_all()
            assert e.value.status == 1
        else:
            compare(g, og, t.numpy(), [2], 4, 1, block, block)
    g.close()


@pytest.mark.parametrize("shift", [1, 2])
def test_targets_at_any_device_address(cuda_device, shift):
    """Device targets that are not aligned to their four bytes go through a copy."""
    block = 1 << 14
    g, og, *_ = _graph(5000, 8, 16, 9, block)
    t = _targets(5000, 2, 70, 9)
    raw = torch.zeros(t.numel() * 4 + 8, dtype=torch.uint8, device=cuda_device)
    raw[shift:shift + t.numel() * 4] = t.contiguous().view(torch.uint8).flatten().to(cuda_device)
    g.prepare(t.to(cuda_device), [3, 2], 4, 0)
    fan = (ctypes.c_int32 * 2)(3, 2)
    stream = torch.cuda.current_stream().cuda_stream or None
    assert lib().agnes_prepare_hyperbatch(g._ctx, raw.data_ptr() + shift, 2, 70, fan, 2, 5, 0,
                                          stream) == 0
    compare(g, og, t.numpy(), [3, 2], 5, 0, block, block)
    g.close()


@pytest.mark.parametrize("H,B,kind", [(1, 16, "dup"), (2, 100, "range"), (4, 64, "dup"),
                                      (1, 300, "dup"), (3, 200, "range"), (1, 5000, "dup")])
def test_bad_targets_leave_no_counts_behind(cuda_device, H, B, kind):
    """A repeated or out-of-range target is reported (5000 repeats: a cell with
    more entries than its tile has ids), and the next hyperbatch is right."""
    N = 20_000
    g, og, *_ = _graph(N, 8, 16, 4, 1 << 14)
    good = _targets(N, H, B, 1)
    bad = good.clone()
    if kind == "dup":
        bad[H - 1, :] = int(bad[H - 1, 0]) if B == 5000 else bad[H - 1, :]
        bad[H - 1, B - 1] = bad[H - 1, 0]
    else:
        bad[H - 1, B - 1] = N
        bad[0, 0] = -1
    for t in (bad, good, bad, good):
        g.prepare(t.to(cuda_device), [3, 2], 7, 0)
        if t is bad:
            with pytest.raises(AgnesError) as e:
                g.fetch_all()
            assert e.value.status == 1
        else:
            compare(g, og, t.numpy(), [3, 2], 7, 0, 1 << 14, 1 << 14)
    g.close()


@pytest.mark.parametrize("dtype", [torch.float16, torch.float32])
@pytest.mark.parametrize("dim,shift", [(1, 0), (2, 0), (3, 0), (7, 1), (8, 1), (16, 0), (25, 0),
                                       (50, 0), (96, 0), (100, 0), (127, 3), (128, 0), (130, 0),
                                       (256, 0), (301, 0), (602, 2), (1030, 0),
                                       (1024, 0), (1032, 0), (1400, 0), (1408, 0), (2040, 0),
                                       (2048, 0), (2056, 0), (3072, 0)])
def test_rows_of_any_width(cuda_device, dtype, dim, shift):
    """Rows of every alignment, from a matrix that starts `shift` elements past
    an aligned address: the first and last rows are read at the matrix's ends."""
    N = 3000
    off, ind = synth.rmat_csr(N, 5, 0.57, 0.19, 0.19, 8)
    gen = torch.Generator().manual_seed(dim)
    flat = torch.randint(0, 1 << 15, (shift + N * dim,), generator=gen, dtype=torch.int32)
    flat = flat.to(torch.int16).view(torch.float16) if dtype == torch.float16 else \
        flat.view(torch.float32)
    dev = flat.to(cuda_device)
    feats = dev[shift:].view(N, dim)
    g = Graph(off.to(cuda_device), ind.to(cuda_device), feats, adj_block_bytes=1 << 14,
              feat_block_bytes=max(1 << 14, feats.element_size() * dim))
    t = _targets(N, 3, 500, 2)
    t[0, 0], t[0, 1] = 0, N - 1
    t[0, 2:] = torch.arange(1, 499, dtype=torch.int32)
    g.prepare(t.to(cuda_device), [4], 3, 0)
    bits = torch.int16 if dtype == torch.float16 else torch.int32
    for j in range(3):
        v = g.fetch(j)
        assert torch.equal(v.feats.view(bits), feats[v.nodes.long()].view(bits))
    g.close()


@pytest.mark.parametrize("d_in,d_out,dtype,fan,H,B", [
    (8, 32, torch.float16, [3], 1, 5),          # one tile of 32 rows, no swizzle
    (24, 64, torch.float16, [40], 2, 70),       # tiles of 32 rows; 40 neighbours
    (32, 32, torch.float16, [6], 3, 1500),      # one swizzled block of 64 elements
    (96, 96, torch.float32, [7], 2, 2000),      # tiles of 64 rows
    (128, 128, torch.float16, [5], 40, 600),    # tiles of 128 rows, several per CTA
    (160, 64, torch.float16, [9], 4, 400),
    (200, 160, torch.float16, [4], 2, 300),     # the most shared memory, no swizzle
    (360, 32, torch.float32, [3], 2, 200),
    (224, 128, torch.float16, [12], 2, 500),    # one stage, few indices staged
    (64, 256, torch.float16, [300], 2, 60),     # more edges in a tile than are staged
    (64, 64, torch.float16, [4], 256, 3),       # the most minibatches whose tiles travel along
    (64, 64, torch.float16, [4], 257, 3),       # one more: tables on the device
    (96, 32, torch.float16, [200], 6, 8000),    # heavy rows: tiles of 64, the smallest W behind
    (104, 256, torch.float16, [200], 3, 5000),  # the same without swizzle
    (128, 256, torch.float16, [1], 4, 6000),    # light rows, one stage of 128
    (128, 256, torch.float32, [60], 6, 8000),   # heavy ones, two of 64, more tiles than stages
    (8, 32, torch.float16, [30], 8, 25000),     # nothing staged; six stages, all used again
    (24, 64, torch.float16, [5], 8, 15000),     # the last width that is not staged, four
    (16, 32, torch.float32, [9], 8, 25000),     # staged, six stages
])
def test_sage_layer_shapes(cuda_device, d_in, d_out, dtype, fan, H, B):
    N = 30_000
    off, ind = synth.rmat_csr(N, 24, 0.6, 0.2, 0.15, 5)
    feats = synth.normal_features(N, d_in, dtype, 6)
    g = Graph(off.to(cuda_device), ind.to(cuda_device), feats.to(cuda_device),
              adj_block_bytes=1 << 16, feat_block_bytes=1 << 16)
    g.prepare(_targets(N, H, B, 3).to(cuda_device), fan, 2, 0)
    allv = g.fetch_all()
    w, b = _weights(d_in, d_out, 1, cuda_device)
    for out_dtype in (torch.float32, torch.float16):
        out = g.sage_mean_layer(0, allv.feats, w, b, out_dtype=out_dtype)
        _check_layer(allv, 0, allv.feats, w, b, out, dtype == torch.float16,
                     out_dtype == torch.float16)
    g.close()


def test_sage_layer_output_16_byte_aligned(cuda_device):
    """An output that is 16- but not 32-byte aligned, through the C ABI."""
    g, *_ = _graph(5000, 8, 64, 9, 1 << 14)
    t = _targets(5000, 2, 90, 1)
    g.prepare(t.to(cuda_device), [5], 1, 0)
    v = g.fetch_all()
    w, b = _weights(64, 96, 1, cuda_device)
    flat = torch.zeros(8 + 2 * 90 * 96, dtype=torch.float16, device=cuda_device)
    rc = lib().agnes_sage_mean_layer(g._ctx, 0, v.feats.data_ptr(), 1, v.feats.shape[1], 64,
                                     w.data_ptr(), b.data_ptr(), 96, flat.data_ptr() + 16, 1, 90,
                                     ctypes.c_void_p(None))
    assert rc == 0
    ref = g.sage_mean_layer(0, v.feats, w, b, out_dtype=torch.float16)
    assert torch.equal(flat[8:].view(2, 90, 96), ref)
    assert torch.count_nonzero(flat[:8]) == 0
    g.close()
    assert np.isfinite(ref.float().cpu().numpy()).all()


@pytest.mark.parametrize("H,B,shift,out_dtype", [
    (4, 2000, 0, torch.float16),    # out == x
    (4, 2000, 3, torch.float16),    # three rows past x
    (4, 2000, -5, torch.float16),   # five rows before it
    (4, 2000, 0, torch.float32),    # wider rows over the same memory
    (300, 20, 0, torch.float16),    # tiles in tables on the device
])
def test_sage_layer_in_place(cuda_device, H, B, shift, out_dtype):
    """An output that shares memory with x holds what a separate one gets, and
    rows past a minibatch's |dst_0| are not written."""
    d = 64
    g, *_ = _graph(20_000, 16, d, 9, 1 << 14)
    g.prepare(_targets(20_000, H, B, 1).to(cuda_device), [6], 1, 0)
    v = g.fetch_all()
    w, b = _weights(d, d, 1, cuda_device)
    ref = g.sage_mean_layer(0, v.feats, w, b, out_dtype=out_dtype)
    rows, size = v.feats.shape[1], ref.element_size() // 2
    buf = torch.empty(2 * v.feats.numel() + 16 * d, dtype=torch.float16, device=cuda_device)
    x = buf[8 * d:8 * d + v.feats.numel()].view(v.feats.shape)
    x.copy_(v.feats)
    before = buf.clone()
    first = (8 + shift) * d  # out's first element of buf
    rc = lib().agnes_sage_mean_layer(g._ctx, 0, x.data_ptr(), 1, rows, d, w.data_ptr(),
                                     b.data_ptr(), d, buf[first:].data_ptr(), int(out_dtype == torch.float16), rows,
                                     ctypes.c_void_p(None))
    assert rc == 0
    want = before
    for j in range(H):
        at = first + j * rows * d * size
        want[at:at + B * d * size] = ref[j, :B].view(torch.float16).flatten()
    assert torch.equal(buf.view(torch.int16), want.view(torch.int16))
    g.close()


@pytest.mark.parametrize("dtype,fan", [(torch.float16, 45), (torch.float32, 45),
                                       (torch.float16, 3)])
def test_sage_mean_is_the_rounded_quotient(cuda_device, dtype, fan):
    """With W_self = 0 and W_neigh = I the layer returns max(mean, 0) as the
    tensor core's input holds it: bit for bit the neighbours' rows added in
    fp32 in edge order, divided in fp32 (numpy's correctly rounded division)
    and rounded to fp16, over degrees 0 .. fan and magnitudes from fp16's
    subnormals to its largest values."""
    N, H, B, d = 20_000, 2, 1500, 64
    off, ind = synth.rmat_csr(N, 24, 0.6, 0.2, 0.15, 5)
    gen = torch.Generator().manual_seed(fan)
    feats = torch.randn(N, d, generator=gen) * 2.0 ** torch.randint(-24, 14, (N, 1), generator=gen)
    feats = feats.to(dtype)
    g = Graph(off.to(cuda_device), ind.to(cuda_device), feats.to(cuda_device),
              adj_block_bytes=1 << 16, feat_block_bytes=1 << 16)
    g.prepare(_targets(N, H, B, 3).to(cuda_device), [fan], 2, 0)
    v = g.fetch_all()
    w = torch.zeros(d, 2 * d, dtype=torch.float16)
    w[:, d:] = torch.eye(d)
    out = g.sage_mean_layer(0, v.feats, w.to(cuda_device), out_dtype=torch.float16).cpu().numpy()
    x = v.feats.float().cpu().numpy()
    seen = set()
    for j in range(H):
        m = v.view(j)
        ptr, col = m.hops[0].indptr.cpu().numpy(), m.hops[0].col.cpu().numpy()
        deg = (ptr[1:] - ptr[:-1]).astype(np.int64)
        acc = np.zeros((B, d), np.float32)
        for s in range(fan):
            rows = np.nonzero(deg > s)[0]
            acc[rows] += x[j][col[ptr[rows] + s]]
        mean = acc / np.maximum(deg, 1).astype(np.float32)[:, None]
        ref = np.maximum(mean.astype(np.float16), np.float16(0))
        assert np.array_equal(out[j, :B], ref)
        seen.update(deg.tolist())
    assert len(seen) > min(fan, 20)
    g.close()
