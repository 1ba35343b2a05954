"""Failure paths, exercised without faulting the GPU.

Injected attempt failures (a host-side flag) must retry with the next seeds
exactly as a failed peel or an unsolvable system does; and a wait of the
dataflow assignment that nothing can satisfy (no vertex starts final) must
give up after its poll limit, return VF_ETIMEOUT and leave the CUDA context
usable for the next build."""
import numpy as np
import pytest

from paper_2503_18397_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

GEOM = ("regime", "h", "shards", "M", "c", "lg_seg", "seg", "l", "T", "cells", "total_cells", "data_bytes")


@pytest.fixture(scope="module")
def vf():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2503_18397_gb300 import build

    build.build()
    import paper_2503_18397_gb300 as vf

    vf.lib()
    yield vf
    vf.vf_debug_faults()


def _dev(a):
    return torch.from_numpy(a.view(np.int64) if a.dtype == np.uint64 else a).cuda()


def test_injected_failures_retry_with_the_next_seeds(vf, orc):
    n = 1 << 20  # one fuse shard (regime chosen by size, as for the benchmark's 2^20-key VFunc)
    keys, vals = synth.u64_keys(0, n, 61), synth.values(n, 8, 61)
    p = vf.vf_params_default(kind=vf.FUNC, b=8, seed=11)
    try:
        vf.vf_debug_faults(fail_attempts=2)
        s = vf.vf_build(_dev(keys), _dev(vals), params=p)
    finally:
        vf.vf_debug_faults()
    info = s.info
    st, oi, _ = orc.build(orc.default_params(kind=orc.FUNC, b=8, seed=13), keys, vals)
    assert st == orc.OK and oi.retries == 0  # seed 13 succeeds on its own
    assert (info.seed, info.retries, info.regime) == (13, 2, vf.REGIME_FUSE)
    for f in GEOM:
        assert getattr(info, f) == getattr(oi, f), f
    assert (s.query(_dev(keys)).cpu().numpy() == vals).all()
    s.free()
    # more injected failures than retries: the build gives up like any other
    try:
        vf.vf_debug_faults(fail_attempts=3)
        with pytest.raises(vf.VFError) as ei:
            vf.vf_build(_dev(keys), _dev(vals), params=vf.vf_params_default(kind=vf.FUNC, b=8, seed=11,
                                                                            max_retries=2))
        assert ei.value.status == 3  # VF_EBUILD
    finally:
        vf.vf_debug_faults()


def test_assignment_wait_runs_out_and_the_context_stays_usable(vf):
    n = 1 << 20  # one fuse shard: the flow solver and its dataflow assignment
    keys, vals = synth.u64_keys(0, n, 62), synth.values(n, 8, 62)
    p = vf.vf_params_default(kind=vf.FUNC, b=8, seed=5, fuse_solver=vf.SOLVER_FLOW)
    try:
        vf.vf_debug_faults(assign_poll_limit=4096, stall_assign=True)
        with pytest.raises(vf.VFError) as ei:
            vf.vf_build(_dev(keys), _dev(vals), params=p)
        assert ei.value.status == 5  # VF_ETIMEOUT
    finally:
        vf.vf_debug_faults()
    # the same build right after, on the same context
    s = vf.vf_build(_dev(keys), _dev(vals), params=p)
    assert (s.query(_dev(keys)).cpu().numpy() == vals).all()
    s.free()
    torch.cuda.synchronize()


@pytest.mark.parametrize("n,arity,eps", [(1 << 20, 3, 0.001), (5_000_000, 4, 0.01)])
@pytest.mark.parametrize("limit", [1, 10])
def test_exchange_wait_runs_out_and_the_context_stays_usable(vf, limit, n, arity, eps):
    # one shard and several; 4-uniform rounds deal their pushes out, with a barrier of their own
    keys, vals = synth.u64_keys(0, n, 63), synth.values(n, 8, 63)
    p = vf.vf_params_default(kind=vf.FUNC, b=8, seed=7, mode=vf.MODE_FUSE, arity=arity, eps=eps, max_retries=30)
    k, v = _dev(keys), _dev(vals)
    try:
        vf.vf_debug_front(poll_limit=limit)
        for _ in range(3):
            with pytest.raises(vf.VFError) as ei:
                vf.vf_build(k, v, params=p)
            assert ei.value.status == 5  # VF_ETIMEOUT
    finally:
        vf.vf_debug_front()
    s = vf.vf_build(k, v, params=p)
    assert bool((s.query(k) == v).all())
    s.free()
    torch.cuda.synchronize()


@pytest.mark.parametrize("n,arity,eps", [(1 << 20, 3, 0.001), (3_000_000, 3, 0.001), (5_000_000, 4, 0.01),
                                         (9_000_000, 4, 0.001)])
def test_lists_beyond_their_room_go_to_the_worklist(vf, orc, n, arity, eps):
    # the attempt is begun again from the keys: plan, seed and retries as the oracle's, answers exact
    keys, vals = synth.u64_keys(0, n, 64), synth.values(n, 8, 64)
    kw = dict(b=8, seed=9, mode=vf.MODE_FUSE, arity=arity, eps=eps, max_retries=30)
    k, v = _dev(keys), _dev(vals)
    before = vf.vf_peel_attempts()
    try:
        vf.vf_debug_front(list_room=8)
        s = vf.vf_build(k, v, params=vf.vf_params_default(kind=vf.FUNC, **kw))
    finally:
        vf.vf_debug_front()
    info = s.info
    done = [a - b for a, b in zip(vf.vf_peel_attempts(), before)]
    assert done == [0, info.retries + 1, info.retries + 1]
    assert bool((s.query(k) == v).all())
    s.free()
    f = vf.vf_build(k, None, params=vf.vf_params_default(kind=vf.FILTER, **kw))  # by the clusters
    done = [a - b for a, b in zip(vf.vf_peel_attempts(), before)]
    assert done == [f.info.retries + 1, info.retries + 1, info.retries + 1]
    assert (f.info.seed, f.info.retries) == (info.seed, info.retries) and bool(f.query(k).all())
    f.free()
    if n <= 3_000_000:
        st, oi, _ = orc.build(orc.default_params(kind=orc.FUNC, **kw), keys, vals)
        assert st == orc.OK and (oi.seed, oi.retries) == (info.seed, info.retries)
        for g in GEOM:
            assert getattr(info, g) == getattr(oi, g), g
