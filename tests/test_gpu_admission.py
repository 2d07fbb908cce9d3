"""Creating a float32 problem does not wait for the work of other streams (GPU
only): device memory is freed by cudaFree, which waits for the whole device,
so the construction must not free any.  The other streams' work takes 30 ms at
least, a creation or admission about 1 ms."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def pair(w, h, d, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    k = torch.arange(d, device="cuda")
    base = 0.2 + 0.6 * torch.sigmoid((k - 0.4 * d) / 2.0) - 0.5 * torch.sigmoid((k - 0.7 * d) / 3.0)
    s = [(base * (0.3 + torch.rand((h, w, d), generator=g, device="cuda"))).float() for _ in range(2)]
    j, i = torch.meshgrid(torch.arange(h, device="cuda", dtype=torch.float64),
                          torch.arange(w, device="cuda", dtype=torch.float64), indexing="ij")
    return s[0], s[1], j * (w + 4) + i, i * (h + 4) + j


@pytest.mark.parametrize("on_device", [True, False])
@pytest.mark.parametrize("levels", [1, 3])
def test_creation_while_another_stream_evaluates(levels, on_device):
    import paper_2010_06931_gb300 as octmc
    big = octmc.Problem(*pair(256, 256, 256, 1))
    small = pair(40, 36, 47, 2) if on_device else [a.cpu() for a in pair(40, 36, 47, 2)]
    D = torch.zeros(big.disp_shape(0), dtype=torch.float64, device="cuda")
    G = torch.empty_like(D)
    busy, mine = torch.cuda.Stream(), torch.cuda.Stream()
    for st in (busy, mine):  # first use of every kernel
        with torch.cuda.stream(st):
            octmc.Problem(*small, levels=levels).zeros()
    big.eval_objective_grad_async(0, D, G, stream=busy)
    torch.cuda.synchronize()
    for _ in range(250):
        big.eval_objective_grad_async(0, D, G, stream=busy)
    end = torch.cuda.Event()
    end.record(busy)
    with torch.cuda.stream(mine):
        P = octmc.Problem(*small, levels=levels)
    assert not end.query()
    torch.cuda.synchronize()
    assert P.level_shape(0) == (40, 36, 47)


def test_admission_while_another_solve_runs():
    import paper_2010_06931_gb300 as octmc
    kw = dict(gtol=0.0, ftol=0.0)
    octmc.Problem(*pair(40, 36, 48, 2), max_iter=2, **kw).solve_full()  # first use of every kernel
    S = octmc.Server(budget_bytes=16 << 30, max_slots=4)
    long = S.submit(*pair(256, 256, 256, 1), max_iter=400, **kw)
    S.step()
    assert S.state(long) == S.RUNNING
    short = S.submit(*pair(40, 36, 48, 2), max_iter=2, **kw)
    S.step()  # admits it
    S.step()  # retires what has finished
    assert S.state(long) == S.RUNNING
    while S.state(long) != S.DONE or S.state(short) != S.DONE:
        S.step()
    assert S.poll(long)[3] in (0, 1) and S.poll(short)[3] in (0, 1)
