"""GPU parity of stb_layer_stack_resident (a whole list of decode steps as one resident kernel) against the CPU
oracle: every layer of a stack is checked against the oracle fed the same, GPU-produced, input."""
import numpy as np
import pytest

import oracle
import oracle.workloads as wl
import stb_inputs as si

pytestmark = pytest.mark.gpu
TOL = 5e-3


@pytest.fixture(scope="module")
def stb():
    import torch
    assert torch.cuda.is_available()
    from paper_2408_01803_b200 import build
    build.build()
    import paper_2408_01803_b200 as stb
    return stb


def _run(stb, torch, triples, graph=False):
    """Runs the triples (layer, x, out) through the resident kernel; returns (status word, workspace)."""
    steps = stb.make_steps(triples)
    ws = stb.resident_workspace(steps)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    if graph:
        stb.layer_stack_resident(None, ws, dev_status=status, marshalled=steps)      # warm outside capture
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            stb.layer_stack_resident(None, ws, dev_status=status, marshalled=steps)
        for _, _, out in triples:
            out.zero_()
        g.replay()
    else:
        stb.layer_stack_resident(None, ws, dev_status=status, marshalled=steps)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    assert int(ws[:16].view(torch.int32).abs().max().item()) == 0, "the counters at the head of the workspace are not zero after the call"
    return status, ws


def _check_layers(triples, logicals, rows_of=None):
    for k, ((_, x, out), L) in enumerate(zip(triples, logicals)):
        xin = x.double().cpu().numpy()
        got = out.double().cpu().numpy()[:, :L.n]
        if rows_of is None:
            ref = oracle.matmul(oracle.decode(L), xin)
        else:
            rows = rows_of(L.n, k)
            ref = oracle.layer_rows(L, rows, xin)
            got = got[:, rows]
        assert np.abs(got - ref).max() <= TOL * np.abs(ref).max(), k


@pytest.mark.parametrize("batch", [1, 2, 5, 8])
def test_chain_with_per_layer_N(stb, batch):
    """Three chained layers with N = 4, 6, 5 (ragged row counts), then an MLP-shaped tail: gate and up read the same
    input (one phase), down reads gate's fp16 output."""
    import torch
    shapes = [(260, 384, 4), (128, 256 + 128, 6), (100, 128, 5)]      # (n, m, N); m of a layer <= ld of the previous output
    ds = [si.logical_layer(n, m, N, 60 + k, max_salient=9) for k, (n, m, N) in enumerate(shapes)]
    dg = si.logical_layer(200, 384, 6, 71, salient_counts=[1, 17, 32])
    du = si.logical_layer(136, 384, 6, 72, salient_counts=[0, 5, 2])
    dd = si.logical_layer(96, 256, 6, 73)
    layers = [stb.pack_numpy(d) for d in ds + [dg, du, dd]]
    x0 = torch.from_numpy(si.activations(batch, 384, 61)).cuda()
    h1 = torch.zeros(batch, 384, dtype=torch.float16, device="cuda")       # 260 outputs used as 384 inputs: the tail stays 0
    h2 = torch.zeros(batch, 128, dtype=torch.float16, device="cuda")
    y3 = torch.zeros(batch, 100, dtype=torch.float32, device="cuda")
    hg = torch.zeros(batch, 256, dtype=torch.float16, device="cuda")
    hu = torch.zeros(batch, 136, dtype=torch.float32, device="cuda")
    y = torch.zeros(batch, 96, dtype=torch.float32, device="cuda")
    triples = [(layers[0], x0, h1), (layers[1], h1, h2), (layers[2], h2, y3),
               (layers[3], x0, hg), (layers[4], x0, hu), (layers[5], hg, y)]
    _run(stb, torch, triples)
    _check_layers(triples, [oracle.Logical(**d) for d in ds + [dg, du, dd]])
    assert (hg.cpu().numpy()[:, 200:] == 0).all()                            # columns past n untouched


@pytest.mark.parametrize("formats", [(5,), (4, 5, 6)])
@pytest.mark.parametrize("blocks", [1, 15, 17, 33])
def test_row_tiles_of_one_to_sixteen_pieces(stb, blocks, formats):
    """About one row tile per SM, whose tiles are dealt to one warp, to fifteen, and to all sixteen with unequal runs; one row (gathered
    throughout: lists of 5:8 alone have a kernel of their own) and three (the kernel with all forms)."""
    import torch
    n, m = 32 * torch.cuda.get_device_properties(0).multi_processor_count - 5, 128 * blocks
    ds = [si.logical_layer(n, m, N, 1300 + N, max_salient=9) for N in formats]
    layers, Ls = [stb.pack_numpy(d) for d in ds], [oracle.Logical(**d) for d in ds]
    for batch in (1, 3):
        x = torch.from_numpy(si.activations(batch, m, 1310)).cuda()
        triples = [(layer, x, torch.zeros(batch, n, dtype=torch.float32, device="cuda")) for layer in layers]
        _run(stb, torch, triples)
        _check_layers(triples, Ls, rows_of=lambda n, k: np.r_[0:64, n // 2:n // 2 + 32, n - 40:n])


@pytest.mark.parametrize("N,batch", [(4, 1), (5, 1), (5, 8), (6, 1)])
def test_residual_words_are_added_before_the_tiles_of_their_chunk(stb, N, batch):
    """The residual terms of a block, two steps of sixteen with a sum of 1 each, beside one weight's 2^24, where an fp32 sum takes nothing
    less than 2: added to each other first they come through, added to the weight's product they are cut off one after the other."""
    import torch
    n, m = 4096, 11008                                        # a size for gemv_stream_kernel at these rows
    x = np.zeros((batch, m), dtype=np.float16)
    cols = np.arange(0, 128, 8)
    x[:, cols], x[:, cols + 1], x[:, 2] = 1 / 16, 1 / 16, 4096.0
    ngrp, nblk = m // 8, m // 128
    d = {"n": n, "m": m, "N": N, "keep": np.full((n, ngrp), (1 << N) - 1, np.uint8), "sign": np.full((n, ngrp), (1 << N) - 1, np.uint8),
         "region": np.zeros((n, ngrp), np.uint16), "sign2": np.zeros((n, nblk), np.uint32), "salient": np.zeros((nblk, 2), np.uint64),
         "scale": np.empty((n, nblk, 5), np.float16)}
    d["region"][:, :16] = 0xF                                 # block 0: columns 8 g and 8 g + 1 of every group are salient
    d["sign2"][:, 0] = 0xFFFFFFFF
    d["salient"][0] = 0x0303030303030303
    d["scale"][:] = [4096.0, 4096.0, 4096.0, 0.0, 1.0]        # the salient weights are their residual term alone
    d["scale"] = d["scale"].view(np.uint16)
    layer, want = stb.pack_numpy(d), float(2 ** 24 + 2)
    assert layer.info()["status"] == 0
    xd = torch.from_numpy(x).cuda()
    got = {"gemv": stb.gemv(layer, xd)}
    if batch == 1:
        for formats in ((N,), (4, 5, 6)):                     # alone and beside other formats
            other = [stb.pack_numpy(si.logical_layer(64, 128, k, 1400 + k)) for k in formats if k != N]
            small = torch.zeros(1, 128, dtype=torch.float16, device="cuda")
            y = torch.zeros(1, n, dtype=torch.float32, device="cuda")
            _run(stb, torch, [(layer, xd, y)] + [(o, small, torch.zeros(1, 64, dtype=torch.float32, device="cuda")) for o in other])
            got["resident %d formats" % len(formats)] = y
    torch.cuda.synchronize()
    for call, y in got.items():
        assert (y == want).all(), (call, y.unique().tolist())


def test_results_are_reproducible_and_close_to_the_per_layer_launches(stb):
    import torch
    d1, d2 = si.logical_layer(700, 1024, 6, 81, max_salient=12), si.logical_layer(300, 768, 4, 82, max_salient=12)
    l1, l2 = stb.pack_numpy(d1), stb.pack_numpy(d2)
    x = torch.from_numpy(si.activations(2, 1024, 83)).cuda()
    outs = []
    for _ in range(2):
        h = torch.zeros(2, 768, dtype=torch.float16, device="cuda")
        y = torch.zeros(2, 300, dtype=torch.float32, device="cuda")
        _run(stb, torch, [(l1, x, h), (l2, h, y)])
        outs.append((h.clone(), y.clone()))
    assert torch.equal(outs[0][0], outs[1][0]) and torch.equal(outs[0][1], outs[1][1])
    h = torch.zeros(2, 768, dtype=torch.float16, device="cuda")
    y = torch.zeros(2, 300, dtype=torch.float32, device="cuda")
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    stb.layer_stack([(l1, x, h), (l2, h, y)], dev_status=st)
    torch.cuda.synchronize()
    a, b = outs[0][1].double().cpu().numpy(), y.double().cpu().numpy()
    assert np.abs(a - b).max() <= 2e-3 * np.abs(b).max()


def test_more_groups_than_one_launch_holds(stb):
    """70 small steps that alternate between two inputs (no two neighbours can share a group): more than the 64
    groups one launch takes, so the list runs as two launches."""
    import torch
    n = 128
    ds = [si.logical_layer(n, n, 4 + k % 3, 900 + k, max_salient=2) for k in range(4)]
    layers = [stb.pack_numpy(d) for d in ds]
    Ls = [oracle.Logical(**d) for d in ds]
    xs = [torch.from_numpy(si.activations(1, n, 98 + i)).cuda() for i in range(2)]
    outs = [torch.zeros(1, n, dtype=torch.float32, device="cuda") for _ in range(70)]
    triples = [(layers[k % 4], xs[k % 2], outs[k]) for k in range(70)]
    _run(stb, torch, triples)
    _check_layers(triples, [Ls[k % 4] for k in range(70)])


@pytest.mark.parametrize("N,batch,m,rows,steps,counts", [
    (6, 2, 4224, 40, 4, [32, 9, 0, 20]),        # operand-order image, words by their places
    (5, 2, 4224, 3600, 4, [5, 32, 0]),          # plain copy (row tiles read it often enough), words by their places
    (4, 2, 512, 14300, 1, [3, 17]),             # plain copy, words gathered
    (4, 8, 4096, 70, 3, [32, 9, 0, 20]),        # activations through L1, words by their places
    (5, 3, 1408, 5000, 2, [7]),
    (6, 5, 5504, 333, 1, [32]),
    (4, 2, 33024, 64, 1, [2, 0, 32]),           # words too many for their places: by the layer's table
    (5, 1, 12288, 96, 3, [9]),
    (6, 8, 13824, 40, 3, [4]),
])
def test_activations_and_residual_words_in_every_form(stb, N, batch, m, rows, steps, counts):
    """Several layers of one input, and a layer that reads the first one's output: where the activations stand (operand-order
    image, plain copy, global memory) times how the residual words find theirs (gathered, by places, by the layer's table)."""
    import torch
    ds = [si.logical_layer(rows + k, m, N, 1100 + k, salient_counts=counts) for k in range(steps)]
    back = 128 * (rows // 128)
    if back:
        ds.append(si.logical_layer(200, back, 4 + (N - 3) % 3, 1150, salient_counts=[9, 0]))
    layers = [stb.pack_numpy(d) for d in ds]
    x = torch.from_numpy(si.activations(batch, m, 1160)).cuda()
    outs = [torch.zeros(batch, -(-d["n"] // 8) * 8, dtype=torch.float16, device="cuda") for d in ds]
    triples = [(layers[k], x if k < steps else outs[0][:, :back], outs[k][:, :ds[k]["n"]]) for k in range(len(ds))]
    _run(stb, torch, triples)
    _check_layers(triples, [oracle.Logical(**d) for d in ds])


def test_nothing_stays_in_the_workspace(stb):
    """Row tiles that straddle CTAs hand sums on through the workspace: after every call it holds none (nothing but the count of
    launches at its head), so that no sum of an earlier launch can be taken for this one's, however many lie between."""
    import torch
    small, wide = si.logical_layer(320, 4096, 6, 94), si.logical_layer(1000, 2048, 5, 95)
    ls, lw = stb.pack_numpy(small), stb.pack_numpy(wide)
    xs = torch.from_numpy(si.activations(2, 4096, 96)).cuda()
    ys, yw = torch.zeros(2, 320, device="cuda"), torch.zeros(2, 1000, device="cuda")
    lists = [[(ls, xs, ys)], [(lw, xs[:, :2048], yw), (ls, xs, ys)]]
    steps = [stb.make_steps(t) for t in lists]
    ws = torch.zeros(max(stb.resident_workspace(s).numel() for s in steps), dtype=torch.uint8, device="cuda")
    assert ws.numel() > 1024
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    for k in range(4):
        stb.layer_stack_resident(None, ws, dev_status=status, marshalled=steps[k % 2])
        torch.cuda.synchronize()
        assert int(status.item()) == 0 and int(ws[:16].max().item()) == 0 and int(ws[256:].max().item()) == 0
        _check_layers(lists[k % 2], [oracle.Logical(**d) for d in ((small,), (wide, small))[k % 2]])
    stb.layer_stack_resident(None, ws, dev_status=status, marshalled=steps[1], selftest=True)
    torch.cuda.synchronize()
    assert int(status.item()) == stb.STB_ERR_TIMEOUT and int(ws[:16].max().item()) == 0 and int(ws[256:].max().item()) == 0


def test_a_wait_that_runs_out_is_reported_and_the_workspace_is_zero_again(stb):
    import torch
    d1, d2 = si.logical_layer(512, 1024, 6, 91), si.logical_layer(256, 512, 5, 92)
    l1, l2 = stb.pack_numpy(d1), stb.pack_numpy(d2)
    x = torch.from_numpy(si.activations(1, 1024, 93)).cuda()
    h = torch.zeros(1, 512, dtype=torch.float16, device="cuda")
    y = torch.zeros(1, 256, dtype=torch.float32, device="cuda")
    triples = [(l1, x, h), (l2, h, y)]
    steps = stb.make_steps(triples)
    ws = stb.resident_workspace(steps)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    stb.layer_stack_resident(None, ws, dev_status=status, marshalled=steps, selftest=True)
    torch.cuda.synchronize()
    assert int(status.item()) == stb.STB_ERR_TIMEOUT
    assert int(ws[:16].view(torch.int32).abs().max().item()) == 0
    status.zero_()
    stb.layer_stack_resident(None, ws, dev_status=status, marshalled=steps)       # the same workspace, an ordinary call
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    _check_layers(triples, [oracle.Logical(**d1), oracle.Logical(**d2)])


def test_unsupported_steps_are_refused_on_the_host(stb):
    import torch
    d = si.logical_layer(64, 128, 3, 95)
    lay = stb.pack_numpy(d)
    x = torch.zeros(1, 128, dtype=torch.float16, device="cuda")
    y = torch.zeros(1, 64, device="cuda")
    steps = stb.make_steps([(lay, x, y)])
    out = stb.C.c_size_t()
    assert stb._lib.stb_layer_stack_resident_workspace(steps, 1, stb.C.byref(out)) == stb.STB_ERR_UNSUPPORTED      # N = 3
    d4 = si.logical_layer(64, 128, 4, 96)
    lay4 = stb.pack_numpy(d4)
    x9 = torch.zeros(9, 128, dtype=torch.float16, device="cuda")
    y9 = torch.zeros(9, 64, device="cuda")
    steps = stb.make_steps([(lay4, x9, y9)])
    assert stb._lib.stb_layer_stack_resident_workspace(steps, 1, stb.C.byref(out)) == stb.STB_ERR_UNSUPPORTED      # batch 9
    steps = stb.make_steps([(lay4, x, y)])
    ws = stb.resident_workspace(steps)
    assert stb._lib.stb_layer_stack_resident(steps, 1, stb._ptr(ws), 16, None, stb._stream()) == stb.STB_ERR_SIZE


def _check_gated_mlp(stb, torch, dg, du, dd, batch, graph=False, rows_of=None):
    """gate and up read x, down reads fp16(silu(gate) * up) formed while it stages its input (STB_IN_SILU_MUL): gate and
    up against the oracle as usual, down against the oracle fed the oracle's own float64 evaluation of the gated
    activation of the GPU's gate and up outputs."""
    m, f = dg["m"], dg["n"]
    lg, lu, ld = (stb.pack_numpy(d) for d in (dg, du, dd))
    x = torch.from_numpy(si.activations(batch, m, 74)).cuda()
    hg = torch.zeros(batch, f, dtype=torch.float16, device="cuda")
    hu = torch.zeros(batch, f, dtype=torch.float16, device="cuda")
    y = torch.zeros(batch, dd["n"], dtype=torch.float32, device="cuda")
    triples = [(lg, x, hg), (lu, x, hu), (ld, (hg, hu), y)]
    _run(stb, torch, triples, graph=graph)
    as_l = wl.as_logical
    _check_layers(triples[:2], [as_l(dg), as_l(du)], rows_of=rows_of)
    act = oracle.silu_mul(hg.double().cpu().numpy(), hu.double().cpu().numpy())
    got = y.double().cpu().numpy()
    if rows_of is None:
        ref = oracle.matmul(oracle.decode(as_l(dd)), act)
    else:
        rows = rows_of(dd["n"], 2)
        ref = oracle.layer_rows(as_l(dd), rows, act)
        got = got[:, rows]
    assert np.abs(got - ref).max() <= TOL * np.abs(ref).max()


@pytest.mark.parametrize("N,batch", [(6, 1), (6, 2), (6, 3), (4, 1), (5, 8)])
def test_gated_activation_is_formed_while_down_stages_its_input(stb, N, batch):
    import torch
    dg = si.logical_layer(384, 256, N, 171, max_salient=9)
    du = si.logical_layer(384, 256, N, 172, max_salient=9)
    dd = si.logical_layer(200, 384, N, 173, salient_counts=[3, 17, 0])
    _check_gated_mlp(stb, torch, dg, du, dd, batch)


@pytest.mark.parametrize("N,batch,f", [(4, 1, 35456), (6, 1, 24576), (6, 2, 16640), (5, 8, 2560)])
def test_gated_activation_that_fills_shared_memory(stb, N, batch, f):
    """Formed inputs so wide that the activations behind the residual words have no room beside them (the widest, and in between)."""
    import torch
    dg = si.logical_layer(f, 128, N, 175, max_salient=9)
    du = si.logical_layer(f, 128, N, 176, max_salient=9)
    dd = si.logical_layer(70, f, N, 177, salient_counts=[3, 17, 0, 32])
    _check_gated_mlp(stb, torch, dg, du, dd, batch)


@pytest.mark.parametrize("N,batch,f", [(4, 4, 11264), (5, 8, 3840), (6, 4, 8192), (6, 2, 18688), (5, 2, 21760), (4, 1, 40960)])
def test_gated_activation_beside_slots_for_few_residual_words(stb, N, batch, f):
    """Formed inputs that fit only where ring slots hold eight residual words at most: blocks of 32 salient columns then come one
    by one, others in pairs."""
    import torch
    dg = si.logical_layer(f, 128, N, 178, max_salient=9)
    du = si.logical_layer(f, 128, N, 179, max_salient=9)
    dd = si.logical_layer(70, f, N, 180, salient_counts=[32, 32, 3, 17, 0, 9])
    _check_gated_mlp(stb, torch, dg, du, dd, batch)


def _picking_layer(m):
    """A 4:8 layer whose row r is 1 in column r and 0 elsewhere: its output is its staged input."""
    c = np.arange(m)
    keep = np.full((m, m // 8), 0x0F, dtype=np.uint8)
    keep[c, c // 8] = np.where(c % 8 < 4, 0x0F, 0xF0)
    region = np.full((m, m // 8), 0x55, dtype=np.uint16)
    region[c, c // 8] = 0x55 & ~(1 << (2 * (c % 4)))
    scale = np.zeros((m, m // 128, 5), dtype=np.float16)
    scale[..., 0] = 1.0
    return dict(n=m, m=m, N=4, keep=keep, sign=np.full((m, m // 8), 0x0F, dtype=np.uint8), region=region, sign2=np.zeros((m, m // 128), dtype=np.uint32),
                salient=np.zeros((m // 128, 2), dtype=np.uint64), scale=scale.view(np.uint16))


def _formed(stb, torch, gate, up):
    """fp16(silu(gate) * up) as the resident kernel stages it, for arrays of rows of up to 8 x m values."""
    rows, m = gate.shape
    layer, y = stb.pack_numpy(_picking_layer(m)), torch.zeros(rows, m, device="cuda")
    _run(stb, torch, [(layer, (torch.from_numpy(gate).cuda(), torch.from_numpy(up).cuda()), y)])
    return y.cpu().numpy()


@pytest.mark.parametrize("up", [1.0, -0.4375])
def test_gated_activation_of_every_finite_gate(stb, up):
    """All finite fp16 gates against float64: fp32 arithmetic (__expf: 2 + 1.173 |a| ulp; sum, quotient and product another 4), one
    rounding to fp16."""
    import torch
    codes = np.arange(65536, dtype=np.uint16).view(np.float16)
    codes = np.where(np.isfinite(codes), codes, np.float16(0)).reshape(4, 8, 2048)
    for gate in codes:
        got = _formed(stb, torch, gate, np.full_like(gate, up)).astype(np.float64)
        a = gate.astype(np.float64)
        with np.errstate(over="ignore"):
            want = a / (1.0 + np.exp(-a)) * up
        bound = np.abs(want) * (2.0 ** -11 + (6.0 + 1.173 * np.abs(a)) * 2.0 ** -23) * (1 + 2.0 ** -9) + 2.0 ** -25
        assert (np.abs(got - want) <= bound).all()


@pytest.mark.parametrize("a", [np.inf, -np.inf, np.nan, 65504.0, -65504.0, -100.0, -88.0])
@pytest.mark.parametrize("b", [2.0, -0.5, 0.0, np.inf])
def test_gated_activation_of_infinite_and_largest_gates(stb, a, b):
    """What fp32 a / (1 + exp(-a)) * b gives, where a linear before it overflowed."""
    import torch
    gate, up = np.zeros((1, 128), dtype=np.float16), np.ones((1, 128), dtype=np.float16)
    gate[0, 37], up[0, 37] = a, b
    with np.errstate(all="ignore"):
        f = np.float32
        want = float((f(a) / (f(1) + np.exp(f(-a))) * f(b)).astype(np.float16))
    got = float(_formed(stb, torch, gate, up)[0, 37])
    assert got == want or (np.isnan(got) and np.isnan(want)), (got, want)


def test_gated_mlp_full_size(stb):
    """The LLaMA-2-7B MLP at 6:8 (quantizer-made) with the gated activation, in a CUDA graph as bench.py runs it."""
    import torch
    dg, du, dd = (wl.quantized_layer(*si.workload_layer(2, nm)) for nm in ("gate", "up", "down"))
    _check_gated_mlp(stb, torch, dg, du, dd, 1, graph=True, rows_of=_rows_of)


def test_per_layer_launches_refuse_formed_inputs(stb):
    import torch
    d = si.logical_layer(64, 128, 4, 97)
    lay = stb.pack_numpy(d)
    a = torch.zeros(1, 128, dtype=torch.float16, device="cuda")
    y = torch.zeros(1, 64, device="cuda")
    steps = stb.make_steps([(lay, (a, a), y)])
    assert stb._lib.stb_layer_stack(steps, 1, None, stb._stream()) == stb.STB_ERR_UNSUPPORTED


def test_checksum_of_the_streamed_bytes(stb):
    """stb_layer_stack_checksum = XOR of the 32-bit words of [tiles offset, used_bytes) of every step's packed buffer;
    a flipped bit in a tile or in a residual record changes it."""
    import torch
    ds = [si.logical_layer(200, 1024, 6, 301, salient_counts=[1, 9, 32, 0]), si.logical_layer(130, 1024, 6, 302, max_salient=5),
          si.logical_layer(96, 256, 4, 303), si.logical_layer(4096, 1024, 5, 304, max_salient=20)]
    layers = [stb.pack_numpy(d) for d in ds]
    x = torch.zeros(1, 1024, dtype=torch.float16, device="cuda")
    x2 = torch.zeros(1, 256, dtype=torch.float16, device="cuda")
    outs = [torch.zeros(1, d["n"], device="cuda") for d in ds]
    steps = stb.make_steps([(layers[0], x, outs[0]), (layers[1], x, outs[1]), (layers[2], x2, outs[2]), (layers[3], x, outs[3])])

    def expected(lay):
        info = lay.info()
        nblk = lay.m // 128
        t0 = (64 + 128 * nblk + 255) // 256 * 256
        words = lay.buf[t0:info["used_bytes"]].cpu().numpy().view(np.uint32)
        return int(np.bitwise_xor.reduce(words))

    sums = stb.layer_stack_checksum(steps)
    torch.cuda.synchronize()
    got = [int(v) & 0xFFFFFFFFFFFFFFFF for v in sums.cpu().numpy()]
    assert got == [expected(l) for l in layers]
    # one flipped bit in the last byte a pass streams (a residual record), one in the first tile
    for lay, off in ((layers[0], layers[0].info()["used_bytes"] - 1), (layers[3], (64 + 128 * 8 + 255) // 256 * 256 + 5)):
        before = expected(lay)
        lay.buf[off] ^= 0x10
        after = stb.layer_stack_checksum(steps)
        torch.cuda.synchronize()
        k = layers.index(lay)
        assert (int(after[k].item()) & 0xFFFFFFFFFFFFFFFF) == expected(lay) != before
        lay.buf[off] ^= 0x10


def _rows_of(n, k):
    g = np.random.default_rng(1000 + k)
    return np.unique(np.concatenate([[0, 31, 32, n - 1], g.choice(n, 60, replace=False)])).astype(np.int32)


@pytest.mark.parametrize("batch", [1, 8])
def test_7b_decoder_layer_full_size_in_a_graph(stb, batch):
    """The seven linears of a LLaMA-2-7B decoder layer (quantizer-made, N per group of linears from {4, 5, 6}) through
    the resident kernel, captured in a CUDA graph as bench.py runs it."""
    import torch
    h, f = 4096, 11008
    Nq, No, Nm, Nd = (int(v) for v in np.random.default_rng(si.seed_for(5, 1)).choice([4, 5, 6], size=4))
    spec = [("q", Nq), ("k", Nq), ("v", Nq), ("o", No), ("gate", Nm), ("up", Nm), ("down", Nd)]
    ds = []
    for i, (name, N) in enumerate(spec):
        n, m, _, seed = si.workload_layer(5, name, N)
        ds.append(wl.quantized_layer(n, m, N, seed + 64 * i))
    layers = [stb.pack_numpy(d) for d in ds]
    x = torch.from_numpy(si.activations(batch, h, si.seed_for(5, 9))).cuda()
    q, k, v, o = (torch.zeros(batch, h, dtype=torch.float16, device="cuda") for _ in range(4))
    gate, up = (torch.zeros(batch, f, dtype=torch.float16, device="cuda") for _ in range(2))
    y = torch.zeros(batch, h, dtype=torch.float32, device="cuda")
    io = [(x, q), (x, k), (x, v), (q, o), (o, gate), (o, up), (gate, y)]
    triples = [(layers[i], io[i][0], io[i][1]) for i in range(7)]
    _run(stb, torch, triples, graph=True)
    _check_layers(triples, [wl.as_logical(d) for d in ds], rows_of=_rows_of)


def test_mlp_6of8_and_13b_block_full_size(stb):
    """The benchmark's MLP pass (6:8, gate and up as one phase, down on gate's output) and the 13B decoder block at 5:8,
    quantizer-made layers, batch 1."""
    import torch
    ds = [wl.quantized_layer(*si.workload_layer(2, nm)) for nm in ("gate", "up", "down")]
    layers = [stb.pack_numpy(d) for d in ds]
    x = torch.from_numpy(si.activations(1, 4096, si.seed_for(2, 8))).cuda()
    hg, hu = (torch.zeros(1, 11008, dtype=torch.float16, device="cuda") for _ in range(2))
    y = torch.zeros(1, 4096, dtype=torch.float32, device="cuda")
    triples = [(layers[0], x, hg), (layers[1], x, hu), (layers[2], hg, y)]
    _run(stb, torch, triples, graph=True)
    _check_layers(triples, [wl.as_logical(d) for d in ds], rows_of=_rows_of)
    h, f = 5120, 13824
    names = ["q", "k", "v", "o", "gate", "up", "down"]
    ds = [wl.quantized_layer(*si.workload_layer(3, nm)) for nm in names]
    layers = [stb.pack_numpy(d) for d in ds]
    x = torch.from_numpy(si.activations(1, h, si.seed_for(3, 8))).cuda()
    q, k, v, o = (torch.zeros(1, h, dtype=torch.float16, device="cuda") for _ in range(4))
    gate, up = (torch.zeros(1, f, dtype=torch.float16, device="cuda") for _ in range(2))
    y = torch.zeros(1, h, dtype=torch.float32, device="cuda")
    io = [(x, q), (x, k), (x, v), (q, o), (o, gate), (o, up), (gate, y)]
    triples = [(layers[i], io[i][0], io[i][1]) for i in range(7)]
    _run(stb, torch, triples)
    _check_layers(triples, [wl.as_logical(d) for d in ds], rows_of=_rows_of)
