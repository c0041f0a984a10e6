"""Launches that overlap the end of the kernel before them: each call after a
kernel that lets its successor start long before it writes the call's inputs,
on two streams at once, and captured in a graph."""

import ctypes
import os
import subprocess

import pytest
import torch

from paper_2607_13205_gb300 import build as B
from paper_2607_13205_gb300 import inputs as I
from paper_2607_13205_gb300 import rolekv as R

pytestmark = pytest.mark.gpu

DEV = "cuda"

# Eight CTAs that release the next kernel, wait 100 us (at most 1e6 polls of
# the clock) and only then copy src to dst, 16 bytes an access.
WRITER = r"""
#include <cstdint>
__global__ void late_copy(const uint4* src, uint4* dst, long n) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  uint64_t t0, t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t0));
  for (int i = 0; i < 1000000; ++i) {
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    if (t - t0 > 100000) break;
  }
  for (long x = blockIdx.x * 256L + threadIdx.x; x < n; x += 8 * 256L) dst[x] = src[x];
}
extern "C" int launch_late_copy(const void* src, void* dst, long bytes, void* stream) {
  late_copy<<<8, 256, 0, static_cast<cudaStream_t>(stream)>>>(static_cast<const uint4*>(src), static_cast<uint4*>(dst),
                                                             bytes / 16);
  return cudaGetLastError();
}
"""


@pytest.fixture(scope="module")
def late_copy(tmp_path_factory):
    d = tmp_path_factory.mktemp("late")
    src, so = os.path.join(d, "late.cu"), os.path.join(d, "late.so")
    with open(src, "w") as f:
        f.write(WRITER)
    subprocess.run([B.nvcc_path(), *B.ARCH, "-O2", "-shared", "-Xcompiler", "-fPIC", "-o", so, src], check=True)
    fn = ctypes.CDLL(so).launch_late_copy
    fn.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_long, ctypes.c_void_p]

    def call(src, dst):
        assert src.numel() * src.element_size() % 16 == 0
        assert fn(src.data_ptr(), dst.data_ptr(), src.numel() * src.element_size(),
                  torch.cuda.current_stream().cuda_stream) == 0
    return call


class Case:
    """Inputs of every call for one small batch, and the calls, each with the
    input that the kernel just before it writes."""

    def __init__(self, seed, n=3001, L=2):
        w = I.Workload("order", "snapkv", L, 1, 8, 4, 128, n, 32, 7, (0.25,), 4, (3, 5), (1, 3))
        self.w, self.bud = w, 0.25
        roles = I.workload_roles(w, seed)
        self.roles = torch.as_tensor(roles, device=DEV)
        self.k, self.v = I.make_kv(w, roles, seed, device=DEV)
        self.qw = I.make_q_window(w, seed, device=DEV)
        self.qd = I.make_q_decode(w, seed, device=DEV)
        self.batch = R.Batch(w.L, w.b, w.Hq, w.Hkv, w.d, w.n)
        g = torch.Generator(device=DEV).manual_seed(seed)
        self.lse = 5.0 + torch.rand(w.L, w.b, w.Hq, w.W, generator=g, device=DEV)
        self.scores = torch.rand(self.batch.score_shape(), generator=g, device=DEV)
        self.params = R.select_params(self.bud, I.PAPER_ALPHA, alpha_key=0.02, key_role=I.ROLE_KEY)
        self.ws = R.workspace(R.OP_COMPRESS, self.batch, w.W)
        self.dws = R.decode_workspace(self.batch, self.bud)
        self.dws_full = R.decode_workspace(self.batch, 1.0)
        self.idx = self.select()

    def select(self):
        idx = torch.empty(self.batch.kept_shape(self.bud), dtype=torch.int32, device=DEV)
        R.role_alloc_select(self.batch, self.scores, self.roles, self.params, idx, pool_k=3)
        return idx

    def score(self):
        sc = torch.empty(self.batch.score_shape(), device=DEV)
        return R.snapkv_score(self.batch, self.qw, self.k, self.w.W, 7, sc, lse_win=self.lse, ws=self.ws)

    def score_two_pass(self):
        sc = torch.empty(self.batch.score_shape(), device=DEV)
        return R.snapkv_score(self.batch, self.qw, self.k, self.w.W, 7, sc, ws=self.ws)

    def quest(self):
        return R.quest_score(self.batch, self.qw, self.k, self.w.W, 16,
                             torch.empty(self.batch.score_shape(), device=DEV))

    def compact(self):
        out = [torch.empty(R.compact_shape(self.batch, self.bud), dtype=torch.bfloat16, device=DEV) for _ in "kv"]
        return torch.stack(R.kv_compact(self.batch, self.k, self.v, self.idx, self.bud, *out))

    def decode(self):
        # the first rows of K and V as a kept cache
        m = R.kept_rows(self.w.n, self.bud)
        out = torch.empty((self.w.L, self.w.b, self.w.Hq, self.w.d), device=DEV)
        return R.decode_attention(self.batch, self.qd, self.k[:, :, :, :m], self.v[:, :, :, :m], self.idx, self.bud,
                                  out, ws=self.dws)

    def decode_full(self):
        out = torch.empty((self.w.L, self.w.b, self.w.Hq, self.w.d), device=DEV)
        return R.decode_attention(self.batch, self.qd, self.k, self.v, None, 1.0, out, compacted=False,
                                  ws=self.dws_full)

    def compress(self):
        idx = torch.empty(self.batch.kept_shape(self.bud), dtype=torch.int32, device=DEV)
        kv = torch.empty((2,) + R.compact_shape(self.batch, self.bud), dtype=torch.bfloat16, device=DEV)
        R.rolekv_compress(self.batch, self.qw, self.k, self.v, self.w.W, 7, self.roles, self.params, idx, kv[0], kv[1],
                          self.ws)
        return kv

    def all(self):
        return [f() for f in (self.select, self.score, self.score_two_pass, self.quest, self.compact, self.decode,
                              self.decode_full, self.compress)]


# (call, the input written late): its stale contents are in range, and wrong
LATE = [("select", "scores"), ("score", "lse"), ("score", "k"), ("quest", "k"), ("quest", "qw"), ("compact", "idx"),
        ("compact", "v"), ("decode", "idx"), ("decode", "qd"), ("decode_full", "k"), ("compress", "k"),
        ("compress", "v")]


@pytest.mark.parametrize("shape", [(3001, 2), (20001, 2), (45003, 2), (45003, 20)],
                         ids=["one", "cluster", "cluster_long", "stream"])
def test_after_a_kernel_that_releases_early(late_copy, shape):
    """The selector's three routes and, on the shortest rows, every call."""
    c = Case(1, *shape)
    for call, name in LATE if shape[0] == 3001 else LATE[:1]:
        buf = getattr(c, name)
        want = getattr(c, call)()
        for _ in range(3):
            good = buf.clone()
            buf.copy_(torch.full_like(good, -1) if name == "idx" else -good)
            torch.cuda.synchronize()
            late_copy(good, buf)
            got = getattr(c, call)()
            torch.cuda.synchronize()
            assert torch.equal(buf, good)
            assert torch.equal(got.view(torch.uint8), want.view(torch.uint8)), (call, name)


@pytest.mark.parametrize("shape", [(3001, 2), (45003, 2)], ids=["one", "cluster"])
def test_two_streams(shape):
    cases = [Case(2, *shape), Case(3, *shape)]
    want = [c.all() for c in cases]
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in cases]
    got = [[], []]
    for _ in range(5):
        for i, c in enumerate(cases):
            with torch.cuda.stream(streams[i]):
                got[i].append(c.all())
    torch.cuda.synchronize()
    for i in range(2):
        for r in got[i]:
            for a, b in zip(r, want[i]):
                assert torch.equal(a.view(torch.uint8), b.view(torch.uint8))


@pytest.mark.parametrize("shape", [(3001, 2), (45003, 2)], ids=["one", "cluster"])
def test_captured_calls_in_a_row(shape):
    c, other = Case(4, *shape), Case(5, *shape)
    want = [c.all(), other.all()]
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        got = c.all()
    names = ("roles", "k", "v", "qw", "qd", "lse", "scores", "idx")
    mine = [getattr(c, x).clone() for x in names]
    for inputs, ref in ((other, want[1]), (c, want[0])):
        src = [getattr(other, x) for x in names] if inputs is other else mine
        for x, t in zip(names, src):
            getattr(c, x).copy_(t)
        for _ in range(3):
            g.replay()
        torch.cuda.synchronize()
        for a, b in zip(got, ref):
            assert torch.equal(a.view(torch.uint8), b.view(torch.uint8))


@pytest.mark.parametrize("call", ["score", "h2o", "decode"])
def test_own_workspace_on_another_stream(call, monkeypatch):
    """A call on a stream of its own without a workspace: what the call
    allocates is not handed out to the current stream while the call may still
    run."""
    c = Case(6)
    qf = I.make_q_full(c.w, 6, device=DEV)
    kept = []
    for name in ("workspace", "decode_workspace"):
        make = getattr(R, name)
        monkeypatch.setattr(R, name, lambda *a, make=make, **k: kept.append(make(*a, **k)) or kept[-1])
    s = torch.cuda.Stream()
    out = torch.empty(c.batch.score_shape(), device=DEV)
    o = torch.empty((c.w.L, c.w.b, c.w.Hq, c.w.d), device=DEV)
    torch.cuda.synchronize()
    if call == "score":
        R.snapkv_score(c.batch, c.qw, c.k, c.w.W, 7, out, stream=s)
    elif call == "h2o":
        R.h2o_score(c.batch, qf, c.k, out, stream=s)
    else:
        R.decode_attention(c.batch, c.qd, c.k, c.v, None, 1.0, o, compacted=False, stream=s)
    assert len(kept) == 1
    ptr, size = kept[0].data_ptr(), kept[0].numel()
    kept.clear()                                     # freed, as when the call returns
    later = [torch.empty(size, dtype=torch.uint8, device=DEV) for _ in range(4)]
    assert all(t.data_ptr() != ptr for t in later)
    torch.cuda.synchronize()
