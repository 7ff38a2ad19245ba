"""GPU: the streamed launch gives the three launches' results bit for bit, on
plans at the edges of its chunks, stages, sets and windows, in place, bucket
range by bucket range, and from several streams and threads at once."""
import threading

import numpy as np
import pytest
import torch

from paper_2606_05613_gb300 import build as nb
from paper_2606_05613_gb300 import native as bk

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda:0")
F32, BF16 = torch.float32, torch.bfloat16


@pytest.fixture(scope="module", autouse=True)
def _built():
    nb.build()
    bk.load()


def _plan(dt, kind, K=1):
    """Bucket offsets, in chunks of ch elements (256 threads x 16 vectors)."""
    ch = 16384 if dt == F32 else 32768
    if kind == "tiny":          # shorter than a vector, a stage, a chunk
        sizes = [1, 2, 3, 7, 8, 9, 15, 17, 255, 257, 4097, ch - 1, ch, ch + 1]
    elif kind == "sets":        # a set of 16 chunks, one more, one less; aligned and not
        sizes = [16 * ch, 17 * ch, 15 * ch, 5, 16 * ch + 1, 33 * ch - 3]
    elif kind == "waves":       # more chunks than SMs, the last ones short
        sizes = [401 * ch + 11, 3, 150 * ch, 153 * ch - 1]
    else:                       # "groups": more than 1024 chunks, ragged groups of 512
        sizes = [1025 * ch + 7, 5000, 1536 * ch + 3] if K <= 4 else [5000, 1025 * ch + 7, 3]
    return np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)


def _grads(K, dt, n, seed):
    g = torch.Generator(device=DEV).manual_seed(seed)
    s = torch.randn(n, generator=g, device=DEV)
    return [(torch.randn(n, generator=g, device=DEV) + 0.4 * (-1) ** k * s).to(dt)
            for k in range(K)]


def _params(flag):
    p = bk.bkmoo_default_params()
    p.flags |= flag
    return p


def _run(res, grads, rule, odt, flag, inplace=False, step=0, stream=None):
    g = [x.clone() for x in grads] if inplace else grads
    n, B, K = int(res.offsets[-1]), res.n_buckets, len(g)
    out = g[0] if inplace else torch.full((n,), 3.0, dtype=odt, device=DEV)
    w = torch.full((B, K), -1.0, device=DEV)
    st = torch.full((B,), -1, dtype=torch.int32, device=DEV)
    kw = dict(params=_params(flag), out_weights=w, out_status=st, stream=stream)
    if step:
        for b in range(0, B, step):
            res.resolve_buckets(g, b, min(B, b + step), rule, out, **kw)
    else:
        res.resolve(g, rule, out, **kw)
    return out, w, st


def _same(a, b):
    for x, y in zip(a, b):
        assert torch.equal(x.view(torch.uint8), y.view(torch.uint8))


@pytest.mark.parametrize("kind", ["tiny", "sets", "waves", "groups"])
@pytest.mark.parametrize("dt", [F32, BF16])
@pytest.mark.parametrize("K", range(1, 9))
def test_stream_is_the_three_launches(K, dt, kind):
    off = _plan(dt, kind, K)
    grads = _grads(K, dt, int(off[-1]), 7 * K)
    res = bk.Resolver(K, dt, off, DEV)
    for rule, odt, inplace in (("mgda", dt, False), ("pcgrad", F32, False),
                               ("cagrad", BF16, False), ("mgda", dt, True)):
        three = _run(res, grads, rule, odt, bk.BKMOO_FLAG_THREE_PASS, inplace)
        one = _run(res, grads, rule, odt, bk.BKMOO_FLAG_FUSED, inplace)
        torch.cuda.synchronize()
        assert res.status() == 0
        _same(three, one)
    three = _run(res, grads, "mgda", dt, bk.BKMOO_FLAG_THREE_PASS)
    by_range = _run(res, grads, "mgda", dt, 0, step=3)     # windows inside the plan
    torch.cuda.synchronize()
    assert res.status() == 0
    _same(three, by_range)


def test_stream_nonfinite_and_zero_buckets():
    """NaN, infinities, and zero gradients: the row words' "not written" value
    is no partial's."""
    ch = 16384
    off = np.array([0, 3 * ch, 5 * ch, 9 * ch, 10 * ch], dtype=np.int64)
    grads = _grads(4, F32, int(off[-1]), 3)
    grads[1][ch + 5] = float("nan")
    grads[2].view(torch.int32)[4 * ch] = -1          # the NaN of all ones
    for g in grads:
        g[int(off[2]):int(off[3])] = 0.0
    grads[0][int(off[3])] = float("inf")
    res = bk.Resolver(4, F32, off, DEV)
    for rule in ("mgda", "pcgrad", "cagrad", "mean"):
        three = _run(res, grads, rule, F32, bk.BKMOO_FLAG_THREE_PASS)
        one = _run(res, grads, rule, F32, bk.BKMOO_FLAG_FUSED)
        torch.cuda.synchronize()
        assert one[2].tolist() == [bk.BKMOO_ERR_NONFINITE, bk.BKMOO_ERR_NONFINITE, 0,
                                   bk.BKMOO_ERR_NONFINITE]
        assert res.status() == 0
        _same(three[1:], one[1:])
        _same([three[0][int(off[2]):int(off[3])]], [one[0][int(off[2]):int(off[3])]])
        assert torch.equal(torch.isnan(three[0]), torch.isnan(one[0]))


@pytest.mark.parametrize("shared", [False, True])
def test_stream_from_several_streams_and_threads(shared):
    """Two threads, a stream of another priority each, many resolves at once:
    workspaces of their own, or disjoint bucket ranges of one plan and
    workspace."""
    ch, K = 16384, 4
    off = np.array([0] + [40 * ch * (i + 1) + 13 * i for i in range(6)], dtype=np.int64)
    grads = _grads(K, F32, int(off[-1]), 11)
    ws = [bk.Resolver(K, F32, off, DEV) for _ in range(1 if shared else 2)]
    want = _run(ws[0], grads, "mgda", F32, bk.BKMOO_FLAG_THREE_PASS)
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream(DEV, priority=p) for p in (0, -1)]
    n, B = int(off[-1]), len(off) - 1
    outs = [[torch.zeros(n, device=DEV), torch.zeros(B, K, device=DEV),
             torch.zeros(B, dtype=torch.int32, device=DEV)] for _ in range(1 if shared else 2)]
    torch.cuda.synchronize()
    errors = []

    def work(t):
        try:
            o = outs[0 if shared else t]
            r = ws[0 if shared else t]
            for _ in range(20):
                kw = dict(out_weights=o[1], out_status=o[2], stream=streams[t])
                if shared:
                    r.resolve_buckets(grads, 3 * t, 3 * t + 3, "mgda", o[0], **kw)
                else:
                    r.resolve(grads, "mgda", o[0], params=_params(bk.BKMOO_FLAG_FUSED), **kw)
        except Exception as e:  # noqa: BLE001
            errors.append(e)

    threads = [threading.Thread(target=work, args=(t,)) for t in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not errors
    for r in ws:
        assert r.status() == 0
    for o in outs:
        _same(want, o)


@pytest.mark.parametrize("withhold", [bk.BKMOO_FLAG_TEST_WITHHOLD,
                                      bk.BKMOO_FLAG_TEST_WITHHOLD_EXCHANGE])
@pytest.mark.parametrize("K,dt", [(1, F32), (4, BF16), (8, F32)])
def test_stream_gives_up_inside_a_chunk(K, dt, withhold):
    """A wait that runs out while the other CTAs are several chunks into a
    bucket (their Gram warps leave a chunk unfinished, its tensor-memory stores
    in flight): the call ends with BKMOO_ERR_TIMEOUT, and the next one on the
    same workspace, which takes the same tensor memory, is right."""
    ch = 16384 if dt == F32 else 32768
    off = np.array([0, 700 * ch, 1400 * ch + 5], dtype=np.int64)
    grads = _grads(K, dt, int(off[-1]), K)
    res = bk.Resolver(K, dt, off, DEV)
    want = _run(res, grads, "mgda", dt, bk.BKMOO_FLAG_THREE_PASS)
    _run(res, grads, "mgda", dt, bk.BKMOO_FLAG_FUSED | withhold)
    assert res.status() == bk.BKMOO_ERR_TIMEOUT
    got = _run(res, grads, "mgda", dt, bk.BKMOO_FLAG_FUSED)
    assert res.status() == 0
    _same(want, got)


@pytest.mark.parametrize("step", [0, 3])
def test_withholding_flags_need_the_fused_flag(step):
    """A default call, and one over ranges (which ignores BKMOO_FLAG_FUSED), is
    right whatever the withholding test flags say."""
    off = _plan(F32, "sets")
    grads = _grads(4, F32, int(off[-1]), 2)
    res = bk.Resolver(4, F32, off, DEV)
    want = _run(res, grads, "mgda", F32, bk.BKMOO_FLAG_THREE_PASS)
    flag = bk.BKMOO_FLAG_TEST_WITHHOLD | bk.BKMOO_FLAG_TEST_WITHHOLD_EXCHANGE
    got = _run(res, grads, "mgda", F32, flag | (bk.BKMOO_FLAG_FUSED if step else 0), step=step)
    assert res.status() == 0
    _same(want, got)


@pytest.mark.parametrize("rule", ["mgda", "cagrad"])
@pytest.mark.parametrize("K", [2, 3, 4])
def test_frank_wolfe_alone_is_the_three_launches(K, rule):
    """Without the exact completion the default call (three launches for
    K >= 3, whatever BKMOO_FLAG_FUSED says) gives the three launches' bits."""
    off = _plan(F32, "sets")
    grads = _grads(K, F32, int(off[-1]), 17)
    res = bk.Resolver(K, F32, off, DEV)
    got = []
    for flag in (bk.BKMOO_FLAG_THREE_PASS, 0, bk.BKMOO_FLAG_FUSED):
        p = bk.bkmoo_default_params()
        p.flags = flag
        out = torch.zeros(int(off[-1]), device=DEV)
        w = torch.zeros(res.n_buckets, K, device=DEV)
        st = torch.zeros(res.n_buckets, dtype=torch.int32, device=DEV)
        res.resolve(grads, rule, out, params=p, out_weights=w, out_status=st)
        torch.cuda.synchronize()
        assert res.status() == 0
        got.append((out, w, st))
    _same(got[0], got[1])
    _same(got[0], got[2])


def test_stream_under_graph_capture():
    """Captured once, replayed on new inputs."""
    off = _plan(F32, "sets")
    K = 3
    res = bk.Resolver(K, F32, off, DEV)
    grads = _grads(K, F32, int(off[-1]), 5)
    out = torch.zeros(int(off[-1]), device=DEV)
    s = torch.cuda.Stream(DEV)
    p = _params(bk.BKMOO_FLAG_FUSED)
    res.resolve(grads, "mgda", out, params=p, stream=s)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        res.resolve(grads, "mgda", out, params=p)
    for seed in (21, 22):
        for g, x in zip(grads, _grads(K, F32, int(off[-1]), seed)):
            g.copy_(x)
        graph.replay()
        torch.cuda.synchronize()
        got = out.clone()
        want = _run(res, grads, "mgda", F32, bk.BKMOO_FLAG_THREE_PASS)[0]
        assert torch.equal(got, want)
        assert res.status() == 0


@pytest.mark.parametrize("dt", [F32, BF16])
@pytest.mark.parametrize("K", range(2, 9))
def test_bulk_fed_gram_is_the_register_kernels(K, dt):
    """Plans that take the bulk-fed Gram pass (few chunks; K = 6, 7 always)
    against bkmoo_gram_noalloc, which runs the register kernels: the same
    matrices bit for bit, at chunk, stage and vector edges."""
    ch = 16384 if dt == F32 else 32768
    plans = [[1, 5, 7, 8, 63, 4097, ch - 1, ch, ch + 1, 3 * ch + 9], [100 * ch + 3]]
    if K in (6, 7):
        plans.append([200 * ch, 301 * ch - 5, 17, 111 * ch + 1])
    for sizes in plans:
        off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
        grads = _grads(K, dt, int(off[-1]), K)
        res = bk.Resolver(K, dt, off, DEV)
        got = torch.zeros(len(sizes), K, K, dtype=torch.float64, device=DEV)
        want = torch.zeros_like(got)
        for bad in (None, float("nan"), float("inf")):
            if bad is not None:                  # in a vector, and in a scalar head or tail
                grads[0][int(off[-1]) // 2] = bad
                grads[1][int(off[-1]) - 1] = -bad
            res.gram(grads, got)
            bk.bkmoo_gram_noalloc(grads, off, want)
            torch.cuda.synchronize()
            assert res.status() == 0
            assert torch.equal(torch.isnan(got), torch.isnan(want))
            assert torch.equal(got.nan_to_num(nan=7.0), want.nan_to_num(nan=7.0))
            assert bad is None or not torch.isfinite(got).all()


@pytest.mark.parametrize("K", [2, 8, 10, 12, 15, 16])
def test_solve_pass_at_the_edges_of_its_two_kernels(K):
    """Plans on both sides of the lines between a block and a warp per bucket
    (two buckets per SM; the longest bucket against the number of buckets),
    three launches: weights and directions are those of each bucket resolved
    alone, bit for bit."""
    sms = torch.cuda.get_device_properties(DEV).multi_processor_count
    ch = 16384
    for sizes in ([64] * (2 * sms), [64] * (2 * sms + 1), [64] * (4 * sms) + [2 * sms * ch],
                  [64] * (4 * sms) + [(2 * sms + 1) * ch]):
        off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
        grads = _grads(K, F32, int(off[-1]), K)
        res = bk.Resolver(K, F32, off, DEV)
        out, w, st = _run(res, grads, "mgda", F32, bk.BKMOO_FLAG_THREE_PASS)
        torch.cuda.synchronize()
        assert res.status() == 0 and not st.any()
        for b in (0, 1, len(sizes) // 2, len(sizes) - 1):
            lo, hi = int(off[b]), int(off[b + 1])
            one = bk.Resolver(K, F32, np.array([0, hi - lo]), DEV)
            alone = _run(one, [g[lo:hi] for g in grads], "mgda", F32, bk.BKMOO_FLAG_THREE_PASS)
            assert torch.equal(alone[1][0], w[b]) and torch.equal(alone[0], out[lo:hi])


@pytest.mark.parametrize("dt", [F32, BF16])
@pytest.mark.parametrize("K", [1, 2, 3, 4, 5])
def test_combination_kernels_at_the_edges_of_their_rule(K, dt):
    """Windows of as many chunks as SMs and one more, and the most chunks whose
    gradients are 192 MiB and one more: the combination of the three launches
    (last chunk first up to K = 4 fp32 and K = 3 bf16) writes the streamed
    launch's bits, fp32 and bf16 out, in place too."""
    sms = torch.cuda.get_device_properties(DEV).multi_processor_count
    ch = 16384 if dt == F32 else 32768
    most = (192 << 20) // (K * 65536)
    for n in (sms, sms + 1, most, most + 1):
        sizes = [ch + 9] * 3 + [(n - 8) * ch - 5] + [7, 2]       # n chunks, starts off the grid
        off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
        grads = _grads(K, dt, int(off[-1]), n)
        res = bk.Resolver(K, dt, off, DEV)
        for odt, inplace in ((F32, False), (BF16, False), (dt, True)):
            _same(_run(res, grads, "mgda", odt, bk.BKMOO_FLAG_THREE_PASS, inplace),
                  _run(res, grads, "mgda", odt, bk.BKMOO_FLAG_FUSED, inplace))
        assert res.status() == 0


@pytest.mark.parametrize("dt", [F32, BF16])
@pytest.mark.parametrize("K", [5, 8, 9, 12, 13, 16])
def test_combination_of_many_gradients_last_chunk_first(K, dt):
    """Windows of one chunk more than SMs, and of as many (K >= 12 bf16 changes
    kernels), and of short chunks (every K): the direction is that of the
    weights, in place too."""
    sms = torch.cuda.get_device_properties(DEV).multi_processor_count
    ch = 16384 if dt == F32 else 32768
    for sizes in ([ch + 9] * 3 + [(sms - 8) * ch - 5] + [7, 2],
                  [ch + 9] * 3 + [(sms - 7) * ch - 5] + [7, 2],
                  [ch // 2 - 3, 5, ch // 4 + 1] * 40 + [4097] * sms):
        off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
        grads = _grads(K, dt, int(off[-1]), K)
        res = bk.Resolver(K, dt, off, DEV)
        got, w, _ = _run(res, grads, "mgda", F32, 0)   # (2 elements: a singular Gram)
        half = _run(res, grads, "mgda", BF16, 0)[0]
        place = _run(res, grads, "mgda", dt, 0, inplace=True)[0]
        assert res.status() == 0
        for b in range(len(sizes)):
            lo, hi = int(off[b]), int(off[b + 1])
            want = torch.zeros(hi - lo, dtype=torch.float64, device=DEV)
            size = torch.zeros_like(want)
            for k in range(K):
                x = grads[k][lo:hi].double() * w[b, k].double()
                want += x
                size += x.abs()
            # K fp32 multiply-adds in a row
            assert ((got[lo:hi] - want).abs() <= K * 2.0 ** -24 * size).all()
        assert torch.equal(half, got.to(BF16)) and torch.equal(place, got.to(dt))
