"""Parity of the CUDA Parareal (SRDS-style) sampler with the fp64 oracle:
the per-stage miss lists, NFE, hits and iteration count exactly, final latents
within 1e-5 (max-abs relative)."""
import math

import numpy as np
import pytest

import workload as W
from oracle.gmm import make_eps_fn
from oracle.ddim import serial_ddim
from oracle.srds import run_srds

pytestmark = pytest.mark.gpu


def oracle_srds(w, tol=None, thresh=None):
    a, x0, mu = W.inputs(w)
    return run_srds(a, x0, make_eps_fn(a, mu, w.gmm_std), w.tol if tol is None else tol,
                    w.cache_thresh if thresh is None else thresh)


def gpu_srds(w, tol=None, thresh=None, mode="sync"):
    import torch
    from paper_2609_36522_gb300.solver import SrdsSolver, GmmDenoiser
    a, x0, mu = W.inputs(w)
    dev = torch.device("cuda")
    s = SrdsSolver(w.T, w.latent_shape, a, w.tol if tol is None else tol,
                   w.cache_thresh if thresh is None else thresh, batch=w.batch)
    g = GmmDenoiser(torch.from_numpy(mu).to(dev), w.gmm_std, a, s.max_rows)
    eps = torch.empty(s.max_rows, w.D, dtype=torch.float32, device=dev)
    s.init(torch.from_numpy(x0).to(dev))
    stages = []
    if mode == "sync":
        while True:
            out = s.step()
            if out is None:
                break
            stages.append([tuple(int(v) for v in row) for row in out.miss_bt.cpu().numpy()])
            g.eps(out.batch_x_ptr, out.miss_bt_ptr, s.n_miss_dev(), eps)
            s.submit_eps(eps)
    else:
        while True:
            out = s.step_async()
            if out is None:
                break
            bx, mb, nm = out
            g.eps(bx, mb, nm, eps)
            s.submit_eps(eps)
    s.poll()
    res = dict(x_final=s.result().cpu().numpy(), stats=s.stats(), stages=stages)
    s.close()
    g.close()
    return res


def compare_srds(w, orc, gpu):
    misses = [[(b, i) for (b, i, hit, _) in batch if not hit] for batch in orc.batches]
    assert gpu["stages"] == misses
    st = gpu["stats"]
    assert st["iters"] == orc.iters
    assert st["nfe"] == orc.nfe and st["hits"] == orc.hits
    scale = np.abs(orc.x_final).max(axis=1)
    rel = np.abs(gpu["x_final"] - orc.x_final).max(axis=1) / scale
    assert rel.max() <= 1e-5, rel
    return rel


def margins(orc, tol, thresh):
    md = min((abs(dl - thresh) / max(thresh, 1e-30) for batch in orc.batches
              for (_, _, _, dl) in batch if dl is not None), default=np.inf)
    me = min((abs(e - tol) / max(tol, 1e-30) for errs in orc.errs for e in errs if e is not None),
             default=np.inf)
    return md, me


@pytest.mark.parametrize("wname", ["srds", "srds_batched"])
def test_srds_parity(wname):
    w = W.ALL[wname]
    orc = oracle_srds(w)
    md, me = margins(orc, w.tol, w.cache_thresh)
    assert md > 1e-6 and me > 1e-6, (md, me)
    compare_srds(w, orc, gpu_srds(w))


def test_srds_small_and_ragged():
    w = W.TINY.with_(T=30, latent_shape=(3, 7, 9), K=4, sampler="srds", batch=3)
    compare_srds(w, oracle_srds(w), gpu_srds(w))


def test_srds_uncached_exact_after_n_iterations():
    """tol = 0 and no cache hits: N iterations, and the serial DDIM result."""
    w = W.SRDS.with_(latent_shape=(4, 16, 16))
    a, x0, mu = W.inputs(w)
    g = gpu_srds(w, tol=0.0, thresh=0.0)
    assert g["stats"]["iters"] == g["stats"]["blocks"] and g["stats"]["hits"] == 0
    serial = serial_ddim(a, x0, make_eps_fn(a, mu, w.gmm_std))[:, -1]
    rel = np.abs(g["x_final"] - serial).max(axis=1) / np.abs(serial).max(axis=1)
    assert rel.max() <= 1e-5, rel


def test_srds_async_equals_sync():
    w = W.SRDS.with_(latent_shape=(4, 16, 16))
    a = gpu_srds(w)
    b = gpu_srds(w, mode="async")
    assert np.array_equal(a["x_final"], b["x_final"])
    assert a["stats"]["nfe"] == b["stats"]["nfe"]


def srds_margin(orc, thresh):
    """The smallest relative distance of an Eq. 4 mean change from tau_cache
    over every hit test of the oracle's run."""
    m = math.inf
    for batch in orc.batches:
        for (_b, _i, _hit, dl) in batch:
            if dl is not None and math.isfinite(dl):
                m = min(m, abs(dl - thresh) / thresh)
    return m


@pytest.mark.parametrize("T,batch,shape,seed", [(1, 2, (4, 4, 4), 31), (2, 1, (4, 8, 8), 31),
                                                (5, 3, (3, 5, 7), 31), (17, 64, (4, 4, 4), 31),
                                                (100, 64, (4, 4, 4), 38)])
def test_srds_edge_shapes(T, batch, shape, seed):
    """Blocks of one step (T = 1, 2: a coarse jump and the fine step of its
    block share a timestep, so the fine stage's new entry feeds the coarse
    stage's distance in the same kernel), ragged blocks and odd D (T = 5), and
    64 trajectories x 5 and x 10 blocks of rows (320 and 640 fine-stage rows:
    more than one wave of planning CTAs, so each CTA narrows several). The
    states behind a hit test differ from the oracle's by the fp32 rounding of
    the denoiser's output, carried through up to T steps and N corrections,
    so a test within a few 1e-6 of tau_cache can go either way (seed 31 at
    T = 100 has one at 6e-6); the cases are seeded with every test at least
    1e-4 away."""
    w = W.TINY.with_(T=T, latent_shape=shape, K=3, sampler="srds", batch=batch, seed=seed)
    orc = oracle_srds(w)
    assert srds_margin(orc, w.cache_thresh) > 1e-4
    compare_srds(w, orc, gpu_srds(w))
    g = gpu_srds(w, mode="async")
    assert g["stats"]["nfe"] == orc.nfe


@pytest.mark.parametrize("shape", [(4, 16, 16), (4, 20, 20), (5, 41, 5), (3, 7, 9)])
def test_srds_row_pieces(shape):
    """The apply kernel's row pieces: exactly one piece of 1024 columns, a
    second piece partly filled (1600), one column past a piece (1025, no
    16-byte rows), a piece of 189 odd columns; and, for the same inputs, eps
    rows that start 4 bytes past a 16-byte boundary (four-byte accesses)
    give the aligned run's latents bit for bit."""
    import torch
    from paper_2609_36522_gb300.solver import SrdsSolver, GmmDenoiser
    w = W.TINY.with_(T=20, latent_shape=shape, K=3, sampler="srds", batch=2, seed=33)
    orc = oracle_srds(w)
    assert srds_margin(orc, w.cache_thresh) > 1e-4
    gpu = gpu_srds(w)
    compare_srds(w, orc, gpu)
    a, x0, mu = W.inputs(w)
    s = SrdsSolver(w.T, w.latent_shape, a, w.tol, w.cache_thresh, batch=w.batch)
    g = GmmDenoiser(torch.from_numpy(mu).cuda(), w.gmm_std, a, s.max_rows)
    eps = torch.empty(s.max_rows * w.D, dtype=torch.float32, device="cuda")
    shifted = torch.empty(s.max_rows * w.D + 1, dtype=torch.float32, device="cuda")[1:]
    s.init(torch.from_numpy(x0).cuda())
    while (out := s.step()) is not None:
        g.eps(out.batch_x_ptr, out.miss_bt_ptr, s.n_miss_dev(), eps)
        shifted.copy_(eps)
        s.submit_eps(shifted)
    s.poll()
    assert np.array_equal(s.result().cpu().numpy(), gpu["x_final"])
    s.close()
    g.close()


@pytest.mark.parametrize("wname", ["srds", "srds_batched"])
def test_srds_generation_graph_equals_host_driven(wname):
    """SrdsSolver.generate through the captured generation (IF nodes, one per
    Parareal iteration; iterations after convergence skipped on the device),
    twice and into a pinned host buffer: x_T, NFE, hits and iterations bit for
    bit those of the host-driven run."""
    import torch
    from paper_2609_36522_gb300.solver import SrdsSolver, GmmDenoiser
    w = W.ALL[wname]
    a, x0, mu = W.inputs(w)
    st = torch.cuda.Stream()
    s = SrdsSolver(w.T, w.latent_shape, a, w.tol, w.cache_thresh, batch=w.batch, stream=st)
    g = GmmDenoiser(torch.from_numpy(mu).cuda(), w.gmm_std, a, s.max_rows, stream=st)
    eps = torch.empty(s.max_rows, w.D, dtype=torch.float32, device="cuda")
    x0d = torch.from_numpy(x0).cuda()
    torch.cuda.synchronize()

    def denoise(bx, mb, nm):
        g.eps(bx, mb, nm, eps)
        return eps

    s.init(x0d)
    while True:
        plan = s.step()
        if plan is None:
            break
        s.submit_eps(denoise(plan.batch_x_ptr, plan.miss_bt_ptr, s.n_miss_dev()))
    want, st_want = s.result().clone(), s.stats()
    host = torch.full((w.batch, w.D), float("nan"), dtype=torch.float32).pin_memory()
    for out in (None, host):
        got = s.generate(x0d, denoise, out=out)
        assert s.generate_path() == "device graph", s.__dict__.get("loop_error")
        assert torch.equal(got.cpu(), want.cpu())
        st_got = s.stats()
        assert (st_got["nfe"], st_got["hits"], st_got["iters"]) == (st_want["nfe"], st_want["hits"], st_want["iters"])
    s.close()
    g.close()


def test_srds_generation_graph_call_order():
    """PA_ERR_STATE: capture_begin not right after pa_srds_init, capture_end
    with nothing open or before every stage was issued (the capture is closed,
    the handle needs pa_srds_init and works after it), launch with nothing
    captured, synchronising calls inside a capture."""
    import torch
    from paper_2609_36522_gb300 import abi
    from paper_2609_36522_gb300.solver import SrdsSolver, GmmDenoiser
    w = W.SRDS
    a, x0, mu = W.inputs(w)
    st = torch.cuda.Stream()
    s = SrdsSolver(w.T, w.latent_shape, a, w.tol, w.cache_thresh, batch=w.batch, stream=st)
    g = GmmDenoiser(torch.from_numpy(mu).cuda(), w.gmm_std, a, s.max_rows, stream=st)
    eps = torch.empty(s.max_rows, w.D, dtype=torch.float32, device="cuda")
    x0d = torch.from_numpy(x0).cuda()
    torch.cuda.synchronize()

    def state_error(f, *args):
        with pytest.raises(abi.PaError) as e:
            f(*args)
        assert e.value.status == abi.PA_ERR_STATE

    state_error(abi.pa_srds_loop_capture_end, s.h)
    state_error(abi.pa_srds_loop_launch, s.h)
    s.init(x0d)
    bx, mb, nm = s.step_async()
    state_error(abi.pa_srds_loop_capture_begin, s.h)     # not right after pa_srds_init
    g.eps(bx, mb, nm, eps)
    s.submit_eps(eps)
    s.init(x0d)
    abi.pa_srds_loop_capture_begin(s.h)
    state_error(abi.pa_srds_loop_capture_begin, s.h)
    state_error(abi.pa_srds_poll, s.h)
    state_error(abi.pa_srds_init, s.h, x0d.data_ptr())
    with torch.cuda.stream(st):
        bx, mb, nm = s.step_async()
        g.eps(bx, mb, nm, eps)
        s.submit_eps(eps)
    state_error(abi.pa_srds_loop_capture_end, s.h)       # stages left: closed, nothing kept
    state_error(abi.pa_srds_loop_launch, s.h)
    s.init(x0d)
    while True:
        plan = s.step()
        if plan is None:
            break
        g.eps(plan.batch_x_ptr, plan.miss_bt_ptr, s.n_miss_dev(), eps)
        s.submit_eps(eps)
    want = s.result().clone()

    def denoise(bx, mb, nm):
        g.eps(bx, mb, nm, eps)
        return eps

    assert torch.equal(s.generate(x0d, denoise), want)
    s.close()
    g.close()


def test_srds_nan_is_not_converged():
    """A NaN in one row of one fine stage: that trajectory's error is NaN from
    then on and it runs to the last iteration, unconverged; the other
    trajectory is the one of a clean run."""
    import torch
    from paper_2609_36522_gb300.solver import SrdsSolver, GmmDenoiser
    w = W.TINY.with_(T=25, latent_shape=(4, 8, 8), K=3, sampler="srds", batch=2, seed=33)
    a, x0, mu = W.inputs(w)

    def run(poison):
        s = SrdsSolver(w.T, w.latent_shape, a, w.tol, w.cache_thresh, batch=w.batch)
        g = GmmDenoiser(torch.from_numpy(mu).cuda(), w.gmm_std, a, s.max_rows)
        eps = torch.empty(s.max_rows, w.D, dtype=torch.float32, device="cuda")
        s.init(torch.from_numpy(x0).cuda())
        stage = 0
        while (out := s.step()) is not None:
            g.eps(out.batch_x_ptr, out.miss_bt_ptr, s.n_miss_dev(), eps)
            if poison and stage == s.blocks + 1:  # iteration 1, its second fine stage
                rows = out.miss_bt[:, 0] == 0
                eps[:out.n_miss][rows.nonzero()[1]] = float("nan")
            s.submit_eps(eps)
            stage += 1
        s.poll()
        res = s.result().cpu().numpy(), s.errors(), s.stats()["iters"], s.blocks
        s.close()
        g.close()
        return res

    clean_x, clean_err, clean_iters, blocks = run(False)
    x, err, iters, _ = run(True)
    assert clean_iters < blocks and iters == blocks
    assert np.isnan(err[:, 0]).all() and np.isnan(x[0]).any()
    assert np.array_equal(x[1], clean_x[1])
    assert np.array_equal(err[:clean_iters, 1], clean_err[:clean_iters, 1])
