"""mtdao_run takes several steps in one launch; the states it leaves are those
of single steps with the averages of the schedule, bit for bit."""
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


def _pair(P, w, M, gdt, count, seed, same_gradient=False):
    """Two handles with the same state under way, and gradients of count steps."""
    engines = [P.MTDAO(w["opt"], M, w["shapes"]) for _ in range(2)]
    gen = torch.Generator(device="cuda").manual_seed(seed)
    n = engines[0].n_padded
    for s in range(engines[0].n_states):
        vals = torch.randn((M, n), device="cuda", generator=gen) * 0.02
        if s == engines[0].n_states - 1:
            vals = vals.abs()
        for e in engines:
            e.state_view(s).copy_(vals)
    shape = (M, n) if same_gradient else (count, M, n)
    g = (torch.randn(shape, device="cuda", generator=gen) * 0.01)
    return engines, g.to(torch.bfloat16) if gdt == "bf16" else g


def _same(a, b):
    torch.cuda.synchronize()
    assert a.t == b.t
    for s in range(a.n_states):
        x, y = a.state_view(s).cpu().numpy(), b.state_view(s).cpu().numpy()
        nan = np.isnan(x)
        assert np.array_equal(nan, np.isnan(y)), s
        assert np.array_equal(x[~nan].view(np.uint32), y[~nan].view(np.uint32)), s


CASES = ([(base, N, gdt, M) for base in ("adam", "adopt", "sgdm") for N in (1, 2, 3, 4)
          for gdt, M in (("f32", 3), ("bf16", 4))]
         + [("adam", 2, "f32", 1), ("adam", 3, "bf16", 2), ("adopt", 4, "f32", 8), ("adam", 4, "f32", 16),
            ("sgdm", 2, "bf16", 16), ("adam", 2, "f32", 17), ("adopt", 1, "bf16", 33)])


@pytest.mark.parametrize("base,N,gdt,M", CASES)
def test_run_equals_single_steps(P, base, N, gdt, M):
    """Periods that fall inside, at the end of and across the launches; 70
    steps need two launches; the first step is single in the original ADOPT
    order (odd N)."""
    px, pu, pv = 5, [3, 7, 4, 70][:N], 6
    w = workload_dict([1000, 7, 4096, 333], M, base=base, betas=(0.9, 0.999, 0.5, 0.99)[:N], px=px, pu=pu,
                      pv=0 if base == "sgdm" else pv, clip="global_norm" if base != "adopt" and N == 2 else "none",
                      rho=0.05, gdt=gdt)
    w["opt"]["adopt_prev_v"] = base == "adopt" and N % 2 == 1
    (a, b), g = _pair(P, w, M, gdt, 70, seed=M * 10 + N)
    lrs = [1e-3 * (1 + k % 3) for k in range(70)]
    a.run(g, lrs)
    for k in range(70):
        b.step(g[k], lrs[k])
    _same(a, b)
    a.run(g[:2], lrs[:2])                          # two steps from an odd count
    for k in range(2):
        b.step(g[k], lrs[k])
    _same(a, b)
    a.close()
    b.close()


@pytest.mark.parametrize("base,prev_v", [("adam", False), ("adopt", False), ("adopt", True), ("sgdm", False)])
def test_run_with_infinite_values(P, base, prev_v):
    """Infinite and NaN gradients inside a run, and infinite states before it:
    an infinite state stays infinite (beta = 0 turns it into NaN)."""
    w = workload_dict([2000], 3, base=base, betas=(0.9, 0.0, 0.99), px=0, pu=0, pv=0)
    w["opt"]["adopt_prev_v"] = prev_v
    (a, b), g = _pair(P, w, 3, "f32", 9, seed=8)
    inf = float("inf")
    for e in (a, b):
        e.t = 5
        for s in range(e.n_states):
            e.state_view(s)[s % 3, 10 * s:10 * s + 3] = torch.tensor([inf, inf if s == e.n_states - 1 else -inf, 1.0],
                                                                     device="cuda")
    g[3, 0, 700], g[4, 1, 701], g[8, 2, 702], g[2, 0, 1500] = inf, -inf, inf, float("nan")
    a.run(g, [1e-3] * 9)
    for k in range(9):
        b.step(g[k], 1e-3)
    _same(a, b)
    a.close()
    b.close()


@pytest.mark.parametrize("M", [4, 24])
def test_run_keeps_anchors_and_reads_one_gradient(P, M):
    """The anchor of an averaged state is its value at the last average, also
    when steps follow it in the same call; one buffer serves every step."""
    w = workload_dict([5000], M, betas=(0.9, 0.999), px=4, pu=3, pv=0)
    (a, b), g = _pair(P, w, M, "f32", 11, seed=M, same_gradient=True)
    for e in (a, b):
        e.track_anchor(0b11)
    a.run(g, [1e-3] * 11)
    for _ in range(11):
        b.step(g, 1e-3)
    _same(a, b)
    for s in (0, 1):
        assert torch.equal(a.pseudo_grad_stats(s), b.pseudo_grad_stats(s))
    a.close()
    b.close()


def test_run_on_gradients_inside_the_states(P):
    """Gradients that are the parameters themselves (the gradient of x^2 / 2):
    every step reads what the one before it wrote."""
    w = workload_dict([3000], 4, betas=(0.9,), px=0, pu=0, pv=0)
    (a, b), _ = _pair(P, w, 4, "f32", 1, seed=3, same_gradient=True)
    a.run(a.state_view(0), [1e-2] * 6)
    for _ in range(6):
        b.step(b.state_view(0), 1e-2)
    _same(a, b)
    a.close()
    b.close()


def test_run_stops_at_a_bad_rate(P):
    w = workload_dict([3000], 4, betas=(0.9,))
    (a, b), g = _pair(P, w, 4, "f32", 6, seed=5)
    with pytest.raises(P.MTDAOError) as e:
        a.run(g, [1e-3, 1e-3, 1e-3, float("nan"), 1e-3, 1e-3])
    assert e.value.code == P.ERR_INVALID
    for k in range(3):
        b.step(g[k], 1e-3)
    _same(a, b)                                    # t counts the steps done
    a.close()
    b.close()


@pytest.mark.parametrize("base,N,gdt,clip", [(base, N, gdt, clip) for base in ("adam", "adopt", "sgdm") for N in (1, 2, 3, 4)
                                             for gdt in ("f32", "bf16") for clip in (False, True)
                                             if not (clip and base == "adopt")])
def test_small_and_large_steps_agree(P, base, N, gdt, clip):
    """Workers together take the step kernel of large states, each of them alone
    that of small ones (up to 28, 54 or 64 warps of 128 elements per SM)."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    most = (28 if base == "sgdm" and N == 1 else 54 if base != "adopt" and N <= 2 else 64) * 128 * sms
    M, numel = 3, most // 2
    w = workload_dict([numel], M, base=base, betas=(0.9, 0.999, 0.5, 0.99)[:N], px=0, pu=[0] * N, pv=0,
                      clip="global_norm" if clip else "none", rho=0.05, gdt=gdt)
    (a, _), g = _pair(P, w, M, gdt, 1, seed=N)
    _.close()
    assert a.n_padded <= most < M * a.n_padded
    small = []
    for m in range(M):
        e = P.MTDAO(w["opt"], 1, w["shapes"])
        for s in range(a.n_states):
            e.state_view(s).copy_(a.state_view(s)[m:m + 1])
        e.step(g[0, m:m + 1], 1e-3)
        small.append(e)
    a.step(g[0], 1e-3)
    for s in range(a.n_states):
        for m in range(M):
            assert torch.equal(a.state_view(s)[m], small[m].state_view(s)[0]), (s, m)
    for e in small + [a]:
        e.close()
