"""Calls of the runtime that fail in the middle of an epoch, made on the host: the library's objects are linked a second
time with a few runtime functions wrapped, a chosen kernel launch returns an error without being made, and what the
library does with its streams after that is counted.  Runs in a child process (a process loads one build); nothing
here faults, traps or hangs the GPU."""
import json
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

pytestmark = pytest.mark.gpu

SHIM = r"""
#include <cuda_runtime.h>
#include <new>
static int fail_at = 0, calls = 0, pending = 0, failed = 0, waits = 0, syncs = 0;
static cudaStream_t own = nullptr;
extern "C" {
// launch number `at` (1-based, 0 = none) from now on fails; events are counted from then on
void shim_arm(int at, void* stream) { fail_at = at; calls = pending = failed = waits = syncs = 0; own = (cudaStream_t)stream; }
int shim_launches() { return calls; }
int shim_waits_of_own() { return waits; }    // waits given to the caller's stream after the failure
int shim_syncs_of_others() { return syncs; }  // other streams waited for on the host after the failure
// operator new number `at` from now on, on this thread, throws
static thread_local int new_at = 0, news = 0;
void shim_arm_new(int at) { new_at = at; news = 0; }
int shim_news() { return news; }
void* __real__Znwm(size_t);
void* __wrap__Znwm(size_t n) {
  if (++news == new_at) throw std::bad_alloc();
  return __real__Znwm(n);
}
cudaError_t __real_cudaLaunchKernelExC(const cudaLaunchConfig_t*, const void*, void**);
cudaError_t __real_cudaGetLastError();
cudaError_t __real_cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned);
cudaError_t __real_cudaStreamSynchronize(cudaStream_t);
cudaError_t __wrap_cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void** a) {
  if (++calls == fail_at) { pending = failed = 1; return cudaErrorLaunchOutOfResources; }
  return __real_cudaLaunchKernelExC(c, f, a);
}
cudaError_t __wrap_cudaGetLastError() {
  if (pending) { pending = 0; return cudaErrorLaunchOutOfResources; }
  return __real_cudaGetLastError();
}
cudaError_t __wrap_cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned f) {
  if (failed && s == own) ++waits;
  return __real_cudaStreamWaitEvent(s, e, f);
}
cudaError_t __wrap_cudaStreamSynchronize(cudaStream_t s) {
  if (failed && s != own) ++syncs;
  return __real_cudaStreamSynchronize(s);
}
}
"""
WRAPPED = ("cudaLaunchKernelExC", "cudaGetLastError", "cudaStreamWaitEvent", "cudaStreamSynchronize", "_Znwm")


def _run(scenario, tmp_path):
    from paper_2012_04930_b200 import build
    build.build()
    shim = tmp_path / "shim.cpp"
    shim.write_text(SHIM)
    objs = []
    for src in build.sources():
        obj = build._object(src, False)
        if not os.path.exists(obj):
            obj = str(tmp_path / (os.path.basename(src) + ".o"))
            subprocess.check_call(["nvcc", *build._flags(False, False), "-c", "-o", obj, src])
        objs.append(obj)
    lib = str(tmp_path / "libgcnsa_wrapped.so")
    subprocess.check_call(["nvcc", *build._ARCH, "-Xcompiler", "-fPIC", "-shared", "-o", lib, str(shim), *objs,
                           *[a for f in WRAPPED for a in ("-Xlinker", f"--wrap={f}")]])
    child = subprocess.run([sys.executable, os.path.abspath(__file__), scenario, lib], capture_output=True, text=True,
                           timeout=300)
    assert child.returncode == 0, child.stderr[-2000:]
    return json.loads(child.stdout.strip().splitlines()[-1])


def _child_build():
    """A build whose k-th host allocation fails, for every k; inputs large enough to go through the upload threads."""
    import numpy as np
    from gen import graphs
    from paper_2012_04930_b200 import gcnsa
    n, f = 20_000, 900
    rowptr, col = graphs.permutation_graph(n, 3, 5)
    x = np.random.default_rng(0).standard_normal((n, f)).astype(np.float32)
    assert x.nbytes + col.nbytes >= 64 << 20
    L, env, codes = gcnsa.lib(), gcnsa.make_env(0), []

    def build():
        return gcnsa.Parts(env, rowptr, col, x, np.zeros(n, np.int32), np.ones(n, np.uint8), 2, 2, 100_000, 3)

    build().close()
    L.shim_arm_new(0)
    build().close()
    total = L.shim_news()
    for at in range(total, 0, -1):
        L.shim_arm_new(at)
        try:
            parts = build()
            codes.append(0)
        except gcnsa.GcnsaError as e:
            codes.append(e.code)
            L.shim_arm_new(0)
            continue
        L.shim_arm_new(0)
        assert np.array_equal(parts.features(0), x[parts.members(0)])
        parts.close()
    print(json.dumps({"total": total, "codes": codes, "oom": gcnsa.ERR_OOM}))


def _child(scenario):
    import numpy as np
    import torch
    from gen import configs
    from paper_2012_04930_b200 import gcnsa
    w = configs.small()
    L, out = gcnsa.lib(), []
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        env = gcnsa.make_env(0)
        parts = gcnsa.Parts(env, w.rowptr, w.col, w.x, w.y, w.train_mask, w.dims[-1], w.m, w.overlap_ppm, w.seed,
                            w.part_mode, w.user_part, w.loss_on_halo)
        if scenario == "sage":
            dims = [w.dims[0], 16, w.dims[-1]]
            ws, wn, bs = configs.sage_weights(dims, 3)
            model = gcnsa.Sage(env, parts, dims, ws, wn, bs, batch=256, batch_graph=0)
            call = model.epoch
        else:
            model = gcnsa.Model(env, parts, w.dims, w.w0, w.b0, lr=w.lr)
            xs = [torch.from_numpy(w.x[parts.members(p)]).pin_memory() for p in range(w.m)]
            loss = np.zeros(1, np.float32)
            call = lambda: model.epoch_host([x.data_ptr() for x in xs], loss)  # noqa: E731
            if scenario == "plain":
                model.close()
                model = gcnsa.Model(env, parts, w.dims, w.w0, w.b0, lr=w.lr, epoch_graph=0)
                call = model.epoch
        call()
        L.shim_arm(0, stream.cuda_stream)
        call()
        total = L.shim_launches()
        for at in (2, total // 3, total // 2, total - (total // 20 if scenario == "sage" else 6)):
            L.shim_arm(at, stream.cuda_stream)
            try:
                call()
                code = 0
            except gcnsa.GcnsaError as e:
                code = e.code
            out.append([code, L.shim_waits_of_own(), L.shim_syncs_of_others()])
            stream.synchronize()
        L.shim_arm(0, stream.cuda_stream)
        call()                       # and the object is usable
        stream.synchronize()
        same = None
        if scenario != "sage":       # as if the failed calls had not been made
            other = gcnsa.Model(env, parts, w.dims, w.w0, w.b0, lr=w.lr, epoch_graph=0)
            for _ in range(3):
                other.epoch()
            same = all(np.array_equal(model.get(what, l), other.get(what, l)) for l in range(2)
                       for what in (gcnsa.GET_W, gcnsa.GET_B, gcnsa.GET_ADAM_M_W, gcnsa.GET_ADAM_V_W))
            other.close()
        model.close()
        parts.close()
    print(json.dumps({"m": w.m, "out": out, "same": same, "err_cuda": gcnsa.ERR_CUDA}))


def test_a_failed_sage_epoch_joins_its_workers(tmp_path):
    """The workers' streams are joined to the caller's however an epoch ends: one wait each after the failure."""
    got = _run("sage", tmp_path)
    for code, waits, _ in got["out"]:
        assert code == got["err_cuda"]
        assert waits == got["m"] - 1


def test_a_failed_epoch_from_host_buffers_reads_them_no_longer(tmp_path):
    """The copies of the caller's buffers have ended when a failed call returns: their stream is waited for."""
    got = _run("host", tmp_path)
    for code, _, syncs in got["out"]:
        assert code == got["err_cuda"]
        assert syncs == 1
    assert got["same"]


def test_an_epoch_that_failed_in_its_passes_can_be_made_again(tmp_path):
    """A launch that fails in the passes of an epoch leaves the parameters, the moments and the step count as they were."""
    got = _run("plain", tmp_path)
    assert [o[0] for o in got["out"]] == [got["err_cuda"]] * 4 and got["same"]


def test_no_host_memory_while_building_is_an_error_code(tmp_path):
    got = _run("build", tmp_path)
    assert got["total"] > 10 and set(got["codes"]) <= {0, got["oom"]} and got["oom"] in got["codes"], got


if __name__ == "__main__":
    if len(sys.argv) == 3:
        from paper_2012_04930_b200 import gcnsa
        gcnsa.use_library(sys.argv[2])
        _child_build() if sys.argv[1] == "build" else _child(sys.argv[1])
