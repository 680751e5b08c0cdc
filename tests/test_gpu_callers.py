"""GPU tests of what a caller may do around the calls: options set for another call, a sharded
step that is dropped, kernels of the caller's own ahead of a step, buffers side by side."""
import ctypes
import subprocess

import pytest
import torch

from paper_2603_18112_gb300 import tula_ags as T
from paper_2603_18112_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2603_18112_gb300 import build
    build.build()
    T.lib()


def _normal_pset(sizes):
    ps = W.ParamSet("sizes")
    for n in sizes:
        ps.add((int(n),), W.KIND_NORMAL)
    return ps


def _workload(seed):
    return W.workload("stress_k4", seed=seed, factor_range=(0.1, 10.0), zero_patterns=False)


@pytest.mark.parametrize("gran", [T.TULA_SCALE_PER_TENSOR, T.TULA_SCALE_PER_ELEMENT])
def test_update_scale_leaves_the_statistics_alone(gran):
    """tula_ags_update_scale with the options of a step, whose layer_stats is set: the rows are
    the step's and stay as they are."""
    wl = _workload(301)
    buf = W.allocate(wl, "cuda", K=2, pset=_normal_pset((1, 5, 1000, 20000)))
    W.fill_state(buf, wl)
    W.fill_grads(buf, wl, step=1)
    elem = [torch.ones_like(t) for t in buf.w]
    st = T.AGSOptimizerStep(buf.w, buf.g, buf.m, scale_elem=elem)
    st.step(wl.lr, wl.momentum, wl.weight_decay)
    rows = st.stats.clone()
    st.hp.granularity = gran
    T.tula_ags_update_scale(buf.g[1], buf.g[0], st.hp)
    torch.cuda.synchronize()
    assert torch.equal(st.stats, rows)
    changed = elem if gran == T.TULA_SCALE_PER_ELEMENT else [st.scale]
    assert all(bool((t != 1).any()) for t in changed)


# Lets its dependents start at once, and writes its output some 300 us later: the way a GEMM with
# programmatic dependent launch may write a weight gradient.
_LATE_WRITER = r"""
__global__ void late_writer(float *dst, const float *src, long long n) {
    asm volatile("griddepcontrol.launch_dependents;");
    unsigned long long t0, t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t0));
    for (int i = 0; i < 100000; ++i) {
        asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
        if (t - t0 > 300000ull) break;
        __nanosleep(500);
    }
    for (long long j = blockIdx.x * (long long)blockDim.x + threadIdx.x; j < n;
         j += (long long)gridDim.x * blockDim.x)
        dst[j] = src[j];
}
extern "C" int write_late(float *dst, const float *src, long long n, void *stream) {
    late_writer<<<64, 256, 0, (cudaStream_t)stream>>>(dst, src, n);
    return (int)cudaGetLastError();
}
"""


@pytest.fixture(scope="module")
def write_late(tmp_path_factory):
    from paper_2603_18112_gb300 import build
    d = tmp_path_factory.mktemp("late_writer")
    (d / "late_writer.cu").write_text(_LATE_WRITER)
    nvcc = build.nvcc_path()
    subprocess.run([nvcc, *build.ARCH, "-shared", "-Xcompiler", "-fPIC", "-cudart", "shared",
                    "-Xlinker", f"-rpath={build.cuda_lib_dir(nvcc)}", str(d / "late_writer.cu"),
                    "-o", str(d / "late_writer.so")], check=True)
    fn = ctypes.CDLL(str(d / "late_writer.so")).write_late
    fn.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_longlong, ctypes.c_void_p]

    def run(dst, src):
        assert dst.numel() == src.numel()
        rc = fn(dst.data_ptr(), src.data_ptr(), dst.numel(),
                torch.cuda.current_stream().cuda_stream)
        assert rc == 0
    return run


@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("call", ["step", "lars", "sharded", "stats", "scale", "scale_elem"])
def test_inputs_written_by_a_kernel_that_lets_its_dependents_start(call, shift, write_late):
    """The caller's kernel just ahead of a call allows programmatic dependent launch and writes the
    gradients after that; the call reads what it has written, bit for bit the results of a call
    made after everything had completed."""
    wl = _workload(331)
    K = 2
    ps = _normal_pset((1, 5, 1000, 30001, 200000))
    elem = [torch.zeros(n, device="cuda") for n in ps.numels]
    runs = []
    for late in (False, True):
        buf = W.allocate(wl, "cuda", K=K, pset=ps, align=1 if shift else 64, shift=shift)
        both = torch.zeros(2 * buf.total, device="cuda")  # every replica in one buffer
        buf.g_flats = [both[:buf.total], both[buf.total:]]
        buf.g = [W._views(f, buf.offsets, ps.shapes, buf.numels) for f in buf.g_flats]
        W.fill_state(buf, wl)
        st = T.AGSOptimizerStep(buf.w, buf.g, buf.m, lars_trust=0.01, scale_elem=elem,
                                rule=T.TULA_RULE_LARS if call == "lars" else T.TULA_RULE_AGS)
        share = st.new_g2_share()
        rows = torch.zeros_like(st.stats)
        for seed_step in (1, 2, 3):
            W.fill_grads(buf, wl, step=seed_step)
            src = both.clone()
            if late:
                both.fill_(3.0)
            torch.cuda.synchronize()
            if late:
                write_late(both, src)
            if call in ("step", "lars"):
                st.step(wl.lr, wl.momentum, wl.weight_decay)
            elif call == "sharded":
                st.shard_reduce(wl.momentum, share)
                st.shard_update(wl.lr, wl.momentum, wl.weight_decay, share)
            elif call == "stats":
                T.tula_layer_stats(buf.w, buf.g, rows, st.workspace)
            else:
                st.hp.granularity = int(call == "scale_elem")
                T.tula_ags_update_scale(buf.g[1], buf.g[0], st.hp)
            torch.cuda.synchronize()
        assert st.error() == 0
        runs.append([both, buf.w_flat, buf.m_flat, st.state, st.stats, st.scale, rows,
                     *(t.clone() for t in elem)])
    for a, b in zip(*runs):
        assert torch.equal(a, b)


@pytest.mark.parametrize("K", [1, 4])
@pytest.mark.parametrize("after", ["sharded", "whole", "stats"])
def test_a_dropped_sharded_step(K, after):
    """Pass 1 of a sharded step whose update never comes (a step dropped for its |G|^2): a step
    taken next on the same workspace -- in two halves or whole, over more tiles than there are
    streaming warps -- has its mean, |G|^2, w and m as if the dropped one had not been, and
    tula_layer_stats takes every tile (|w|^2, which the dropped step has not touched)."""
    wl = _workload(311)
    ps = _normal_pset((6_000_003, 7, 40000, 64))
    runs = []
    for dropped in (False, True):
        buf = W.allocate(wl, "cuda", K=K, pset=ps)
        W.fill_state(buf, wl)
        st = T.AGSOptimizerStep(buf.w, buf.g, buf.m, grid_ctas=1, stats=False)
        share = st.new_g2_share()
        if dropped:
            W.fill_grads(buf, wl, step=1)
            st.shard_reduce(wl.momentum, share)
        W.fill_grads(buf, wl, step=2)
        rows = torch.zeros(ps.n_tensors, T.TULA_STATS_LEN, dtype=torch.float64, device="cuda")
        if after == "sharded":
            st.shard_reduce(wl.momentum, share)
            st.shard_update(wl.lr, wl.momentum, wl.weight_decay, share)
        elif after == "whole":
            st.step(wl.lr, wl.momentum, wl.weight_decay)
        else:
            T.tula_layer_stats(buf.w, buf.g, rows, st.workspace)
        torch.cuda.synchronize()
        assert st.error() == 0
        runs.append([buf.g_flats[0], buf.w_flat, buf.m_flat, st.state, rows[:, T.TULA_STAT_W_SQ]])
    for a, b in zip(*runs):
        assert torch.equal(a, b)


@pytest.mark.parametrize("roles", ["wgm", "mgw", "gwm"])
def test_roles_side_by_side_in_one_buffer(roles):
    """The weights, the gradients and the momentum of each tensor back to back in one buffer, none
    at a 16-byte boundary: the update copies ends of w and m, with whatever shares their 32 bytes,
    while the reduction still writes the mean.  Element by element the results are those of aligned
    buffers, bit for bit."""
    K = 2
    sizes = [1, 2, 3, 5, 6, 7, 9, 11, 13, 127, 2049, 4099, 9217, 20001] * 8
    ps = _normal_pset(sizes)
    wl = _workload(351)
    plain = W.allocate(wl, "cuda", K=K, pset=ps)
    W.fill_state(plain, wl)
    flat = torch.zeros(1 + 4 * sum(sizes), device="cuda")
    views = {"w": [], "g": [[], []], "m": []}
    at = 1
    for n in sizes:
        for role in roles:
            for out in views["g"] if role == "g" else [views[role]]:
                out.append(flat[at:at + n])
                at += n
    assert at == flat.numel()
    for a, b in zip(plain.w, views["w"]):
        b.copy_(a)
    kw = dict(force_branch=T.TULA_BRANCH_SCALED, scale=torch.linspace(0.5, 2.0, len(sizes),
                                                                      device="cuda"))
    steps = [T.AGSOptimizerStep(plain.w, plain.g, plain.m, **kw),
             T.AGSOptimizerStep(views["w"], views["g"], views["m"], **kw)]
    for i in range(4):
        W.fill_grads(plain, wl, step=i)
        for a, b in zip(plain.g, views["g"]):
            for x, y in zip(a, b):
                y.copy_(x)
        for st in steps:
            st.step(wl.lr, wl.momentum, wl.weight_decay)
        torch.cuda.synchronize()
        assert all(st.error() == 0 for st in steps)
        for a, b in ((plain.w, views["w"]), (plain.m, views["m"]), (plain.g[0], views["g"][0])):
            for x, y in zip(a, b):
                assert torch.equal(x, y)
