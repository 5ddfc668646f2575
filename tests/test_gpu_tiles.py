"""The kernels on tiles of all replicas, at the edges of what a tile's width and
threads are chosen by: the fused step (step_sync_wide.cuh) gives the bits of the
step followed by the averages, the average (reduce_kernels.cu) those of
replica_mean.cuh's sums, the diagnostics (stats_wide.cu) the sums in 64 bits; and
of the kernels that take other sizes: the register kernel's blocks an SM, replicas
streamed."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from parity_util import workload_dict

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2510_05361_gb300 as P
    P.load()
    return P


def _pair(P, w, M, gdt, seed, plant=False):
    engines = [P.MTDAO(w["opt"], M, w["shapes"]) for _ in range(2)]
    gen = torch.Generator(device="cuda").manual_seed(seed)
    n = engines[0].n_padded
    for s in range(engines[0].n_states):
        vals = torch.randn((M, n), device="cuda", generator=gen) * 0.02
        if s == engines[0].n_states - 1:
            vals = vals.abs()
        if plant:
            vals[M // 2, 5::97] = float("inf")
            vals[M - 1, 7::89] = float("nan")
            vals[:, 11::83] *= 1e-37                   # differences and their M-th subnormal
            vals[:, 13::79] = vals[M - 1, 13::79]      # equal replicas
            vals[:, 17::73] = -0.0
        for e in engines:
            e.state_view(s).copy_(vals)
    g = torch.randn((M, n), device="cuda", generator=gen) * 0.01
    return engines, g.to(torch.bfloat16) if gdt == "bf16" else g


def _same(a, b):
    for s in range(a.n_states):
        x, y = a.state_view(s), b.state_view(s)
        nan = torch.isnan(x)
        assert torch.equal(nan, torch.isnan(y)), s
        assert torch.equal(x.view(torch.int32).masked_fill(nan, 0), y.view(torch.int32).masked_fill(nan, 0)), s


# (M, numel): one tile, an SM's worth of tiles, tiles of every width; M = 6 to 8
# from 2^20 elements on, most of 5 and 4 from 2^21, of 3 from 2^22; the largest tile set that fits (M = 256, N = 4, f32); above it
CASES = [("adam", 4, "f32", 256, 30000), ("adam", 1, "f32", 256, 512), ("sgdm", 1, "bf16", 256, 1),
         ("adopt", 2, "bf16", 255, 5000), ("adopt", 2, "bf16", 8, 1 << 20), ("sgdm", 3, "f32", 8, (1 << 20) - 256),
         ("adam", 2, "f32", 9, 150000), ("adopt", 1, "f32", 16, 20000), ("sgdm", 2, "bf16", 17, 10001),
         ("adam", 3, "f32", 48, 9999), ("adam", 4, "f32", 64, 9999), ("adopt", 2, "bf16", 64, 9999),
         ("sgdm", 4, "f32", 65, 4999), ("adam", 2, "bf16", 100, 4999), ("adam", 3, "f32", 129, 4999),
         ("adam", 1, "bf16", 257, 3000), ("sgdm", 2, "f32", 6, 1 << 20), ("adopt", 4, "bf16", 7, (1 << 20) + 7),
         ("adam", 3, "f32", 5, (1 << 21) + 3), ("adopt", 2, "bf16", 4, 1 << 21), ("adam", 4, "f32", 3, 1 << 22),
         ("adam", 3, "f32", 5, 7000), ("adopt", 2, "bf16", 6, 7000)]
# M = 5 and ADOPT's M = 6: two blocks an SM or three, by the rounds of the grid
CASES += ([(base, N, gdt, 5, numel) for base, N, gdt in (("adam", 1, "f32"), ("adam", 4, "bf16"), ("adopt", 1, "bf16"),
                                                         ("adopt", 3, "f32"), ("sgdm", 2, "f32"), ("sgdm", 3, "bf16"))
           for numel in (150001, 200003, 300005, 700007)]
          # small and middle states: every form of the means, items dealt out for them
          + [("sgdm", 1, "bf16", M, numel) for M, numel in ((9, 60001), (9, 130001), (10, 180001), (14, 90001), (20, 130001),
                                                            (33, 200), (40, 1500), (64, 5000))]
          + [("sgdm", 3, "f32", 15, 130001), ("sgdm", 3, "f32", 20, 60001), ("adopt", 2, "f32", 9, 60001),
             ("adopt", 4, "bf16", 33, 250), ("adam", 3, "bf16", 24, 2000), ("adam", 1, "f32", 12, 60001)]
          + [("adopt", 1, "f32", 6, 200003), ("adopt", 2, "bf16", 6, 700007), ("adopt", 1, "f32", 5, (1 << 21) + 300)])


@pytest.mark.parametrize("base,N,gdt,M,numel,clip", [c + (clip,) for c in CASES for clip in (False, True)
                                                     if not (clip and c[0] == "adopt")])
def test_fused_tiles_equal_step_then_average(P, base, N, gdt, M, numel, clip):
    w = workload_dict([numel], M, base=base, betas=(0.9, 0.999, 0.5, 0.99)[:N], px=1, pu=1, pv=0 if base == "sgdm" else 1,
                      clip="global_norm" if clip else "none", rho=0.05, gdt=gdt)
    (a, b), g = _pair(P, w, M, gdt, seed=M + N, plant=clip)
    every = (1 << a.n_states) - 1
    for mask in (every, 1, every & ~1, 1 << (a.n_states - 1)):
        a.step(g, 1e-3, mask)
        b.step(g, 1e-3, 0)
        b.sync(mask)
        _same(a, b)
    if not clip:                                       # the last average, against 64 bits
        s = a.n_states - 1
        a.step(g, 1e-3, 0)
        before = a.state_view(s).double()
        a.set_params(a.state_view(0)[0].clone())       # all states but x to zero; v is put back
        a.state_view(s).copy_(before)
        a.t = 5
        a.step(torch.zeros_like(g), 0.0, 1 << s)
        beta = float(w["opt"]["beta2"]) if base != "sgdm" else float(w["opt"]["beta1"][N - 1])
        mean = beta * before.mean(0)
        got = a.state_view(s).double()
        assert bool((got == got[0]).all())
        # the decay rounds each value once (2^-24 of it), the compensated mean a few times
        scale = before.abs().mean(0) + 1e-30
        assert float(((got[0] - mean).abs() / scale).max()) < 4 * 2.0 ** -23
    a.close()
    b.close()


def _mean32(s):
    """replica_mean.cuh in numpy, fp32: [M][n] -> [n]."""
    M, s0 = s.shape[0], s[0]
    parts = []
    for lo, hi in ((1, M // 2), (max(M // 2, 1), M)):
        total = np.zeros_like(s0)
        comp = np.zeros_like(s0)
        for m in range(lo, hi):
            y = (s[m] - s0) - comp
            t = total + y
            comp = (t - total) - y
            total = t
        parts.append(total - comp)
    q = (parts[0] + parts[1]) / np.float32(M)
    mean = np.where(q == 0, s0, s0 + q)
    plain = s0.copy()
    for m in range(1, M):
        plain = plain + s[m]
    return np.where(np.isnan(mean), plain / np.float32(M), mean)


@pytest.mark.parametrize("M,numel", [(14, 3000), (15, 3000), (16, 40000), (32, 20001), (33, 20001), (64, 300),
                                     (100, 3000), (256, 1), (257, 9000), (441, 6000), (1024, 700), (1024, 12000)])
def test_average_on_tiles(P, M, numel):
    w = workload_dict([numel], M, base="sgdm", betas=(0.9,), px=1, pu=1, pv=0)
    (a, b), _ = _pair(P, w, M, "f32", seed=M, plant=True)
    ref = [a.state_view(s).cpu().numpy() for s in range(2)]
    with np.errstate(invalid="ignore", over="ignore"):
        ref = [_mean32(r) for r in ref]
    a.sync(0b11)
    b.sync(0b10)
    for s in range(2):
        got = a.state_view(s).cpu().numpy()
        nan = np.isnan(ref[s])
        assert np.array_equal(np.isnan(got), np.broadcast_to(nan, got.shape)), s
        want = np.broadcast_to(ref[s][~nan], got[:, ~nan].shape)
        assert np.array_equal(got[:, ~nan].view(np.uint32), np.ascontiguousarray(want).view(np.uint32)), s
    x, y = a.state_view(1), b.state_view(1)
    assert torch.equal(x.view(torch.int32).masked_fill(torch.isnan(x), 0), y.view(torch.int32).masked_fill(torch.isnan(y), 0))
    a.close()
    b.close()


@pytest.mark.parametrize("M,numel", [(450, 800001), (600, 200001), (899, 160000), (900, 150001), (1024, 110000)])
def test_streamed_average_equals_tiles(P, M, numel):
    """Many replicas: two states together have columns enough to be streamed, each
    alone is averaged on tiles; the anchor follows."""
    w = workload_dict([numel], M, base="sgdm", betas=(0.9,), px=1, pu=1, pv=0)
    (a, b), _ = _pair(P, w, M, "f32", seed=M, plant=True)
    a.track_anchor(0b10)
    a.sync(0b11)
    b.sync(0b01)
    b.sync(0b10)
    _same(a, b)
    for st in range(2):                                # the anchor is the average
        a.state_view(st).normal_()
    a.sync(0b11)
    change = a.pseudo_grad_stats(1)
    assert float(change[:2 * M + 1].abs().max()) == 0.0 and float(change[2 * M + 1]) > 0.0
    a.close()
    b.close()


@pytest.mark.parametrize("M,numel", [(9, 256), (9, 700001), (12, 200000), (13, 400001), (16, 100), (17, 200001),
                                     (64, 200001), (65, 200001), (128, 5000), (129, 90000), (257, 20000),
                                     (513, 9000), (1024, 8000)])
def test_diagnostics_on_tiles(P, M, numel):
    """One tile a block, runs of several with a shorter last one, every number
    of rows a thread takes, narrow tiles."""
    w = workload_dict([numel], M, base="adam", betas=(0.9,), px=1, pu=1, pv=1)
    (a, b), _ = _pair(P, w, M, "f32", seed=M)
    x0 = torch.randn((a.n_padded,), device="cuda") * 0.1
    x0[numel:] = 0
    keep = [a.state_view(s).clone() for s in range(3)]
    a.set_params(x0)
    a.track_anchor(1)
    for s in range(3):
        a.state_view(s).copy_(keep[s])
        b.state_view(s).copy_(keep[s])
    change = a.pseudo_grad_stats(0)
    stats = a.sync_stats(0b101)
    b.sync(0b101)
    _same(a, b)
    # the anchor is x's average now
    assert float(a.pseudo_grad_stats(0)[: 2 * M + 1].abs().max()) == 0.0

    def close(got, want, scale=None, with_mean=False):
        # A position's four elements are summed in fp32, some 2^-24 off each; the errors
        # are independent, so the sum of numel / 4 of them is good to 2^-24 / sqrt(numel / 4)
        # of the sum of magnitudes.  The mean is rounded where it is added to s_0, which is
        # some sqrt(M) times as large.  Five standard deviations of two such errors.
        tol = 10 * 2.0 ** -24 / max(numel / 4, 1) ** 0.5 * (M ** 0.5 if with_mean else 1.0)
        assert bool(((got - want).abs() <= tol * (want.abs() if scale is None else scale) + 1e-300).all())

    x, anchor = keep[0].double(), x0.double()
    mean = x.mean(0)
    loc, glob = x - anchor, mean - anchor
    close(change[:M], loc.square().sum(1))
    close(change[M:2 * M], (loc * glob).sum(1), (loc * glob).abs().sum(1), True)
    close(change[2 * M], glob.square().sum(), None, True)
    close(change[2 * M + 1], anchor.square().sum())
    for row, s in enumerate((0, 2)):
        v = keep[s].double()
        m = v.mean(0)
        close(stats[row, 0], (v - m).square().sum() / M, None, True)
        close(stats[row, 1], m.square().sum(), None, True)
        close(stats[row, 2:2 + M], v.square().sum(1))
        close(stats[row, 2 + M:], (v * m).sum(1), (v * m).abs().sum(1), True)
    a.close()
    b.close()


@pytest.mark.parametrize("M,numel", [(449, 270001), (450, 262000), (450, 262145), (599, 196607), (599, 393217), (898, 270000),
                                     (899, 81900), (899, 82001), (1024, 98305)])
def test_streamed_diagnostics(P, M, numel):
    """Both sides of the limits above which many replicas are streamed in two passes
    (M = 450 to 599: the change alone)."""
    test_diagnostics_on_tiles(P, M, numel)


@pytest.mark.parametrize("M,numel", [(1, 5), (2, 1024), (3, 2049), (4, 600000), (5, 1100001), (8, 2200003), (7, 4200000)])
def test_register_diagnostics_tiles(P, M, numel):
    """Tiles of 2 to 16 positions per thread, the last one partly filled."""
    test_diagnostics_on_tiles(P, M, numel)


@pytest.mark.parametrize("kind,sizes", [("fused", ((256, 512), (200, 60000))), ("sync", ((1024, 3000), (600, 9000))),
                                        ("stats", ((1024, 3000), (600, 9000)))])
def test_tiles_of_different_sizes_from_two_threads(P, kind, sizes):
    """Two threads, a handle and a stream each, launch the same kernel with tiles of
    different sizes (both above the default limit of shared memory)."""
    import threading
    jobs, errors = [], []
    for M, numel in sizes:
        stream = torch.cuda.Stream()
        w = workload_dict([numel], M, base="adam", betas=(0.9, 0.999, 0.5, 0.99), px=1, pu=1, pv=1)
        e = P.MTDAO(w["opt"], M, w["shapes"], stream.cuda_stream)
        g = torch.zeros((M, e.n_padded), device="cuda")
        out = torch.zeros((e.n_states, 2 + 2 * M), dtype=torch.float64, device="cuda")
        every = (1 << e.n_states) - 1
        run = {"fused": lambda e=e, g=g, every=every: e.step(g, 1e-3, every),
               "sync": lambda e=e, every=every: e.sync(every),
               "stats": lambda e=e, out=out, every=every: P.mtdao_sync_stats(e.h, every, out.data_ptr())}[kind]
        run()
        jobs.append((e, run, stream, g, out))
    torch.cuda.synchronize()
    start = threading.Barrier(len(jobs))

    def work(run, stream):
        try:
            start.wait()
            for k in range(4000):
                run()
                if k % 200 == 199:
                    stream.synchronize()
        except Exception as ex:
            errors.append(ex)

    threads = [threading.Thread(target=work, args=(run, stream)) for _, run, stream, _, _ in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not errors, errors
    for e, *_ in jobs:
        e.close()
