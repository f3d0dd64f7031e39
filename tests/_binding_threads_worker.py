"""Calls the binding from several threads against a stand-in library whose entry point only sleeps and counts how many calls
are inside it at once, on one stream and in all.  Executed as a child process by test_gpu_binding_threads.py, because the
binding keeps the library that it was bound to first.  No kernel is launched; the tensors have to be on a GPU."""
import ctypes
import os
import subprocess
import sys
import tempfile
import threading

STAND_IN = r"""
#include <pthread.h>
#include <stddef.h>
#include <unistd.h>
static pthread_mutex_t m = PTHREAD_MUTEX_INITIALIZER;
static void* stream_of[8];
static int inside[8], streams, all;
int worst_on_a_stream, worst_in_all;
int ssm_scan_fwd_state(void* p, void* x, void* d, void* A, void* B, void* C, void* D, void* z, void* h0, void* out, void* hl,
                       void* sv, void* ws, size_t n, void* stream) {
  pthread_mutex_lock(&m);
  int i = 0;
  while (i < streams && stream_of[i] != stream) ++i;
  if (i == streams) stream_of[streams++] = stream;
  if (++inside[i] > worst_on_a_stream) worst_on_a_stream = inside[i];
  if (++all > worst_in_all) worst_in_all = all;
  pthread_mutex_unlock(&m);
  usleep(3000);
  pthread_mutex_lock(&m);
  --inside[i];
  --all;
  pthread_mutex_unlock(&m);
  return 0;
}
size_t ssm_scan_fwd_workspace_bytes(void* p) { return 4096; }
"""
OTHERS = ("ssm_scan_fwd_fused_dt", "ssm_scan_fwd_static", "ssm_scan_bwd", "ssm_scan_bwd_state", "ssm_scan_bwd_fused_dt",
          "ssm_scan_bwd_fused_dt_state", "ssm_step", "ssm_scan_bwd_workspace_bytes", "ssm_scan_saved_state_bytes",
          "ssm_status_string", "ssm_conv1d_fwd", "ssm_conv1d_bwd", "ssm_conv1d_bwd_workspace_bytes")


def main() -> int:
    import torch
    from paper_2312_00752_b200 import binding as K
    with tempfile.TemporaryDirectory() as d:
        src, lib = os.path.join(d, "stand_in.c"), os.path.join(d, "stand_in.so")
        with open(src, "w") as f:
            f.write(STAND_IN + "".join(f"int {n}(void) {{ return 1; }}\n" for n in OTHERS))
        subprocess.run([os.environ.get("CC", "gcc"), "-shared", "-fPIC", "-o", lib, src, "-lpthread"], check=True)
        native = K._native()
        native.init(lib, K.SsmScanError, torch.OutOfMemoryError)
        counts = ctypes.CDLL(lib)
        dev = torch.device("cuda")
        x = torch.zeros(1, 8, 8, device=dev)
        A, B = torch.zeros(8, 4, device=dev), torch.zeros(1, 8, 4, device=dev)

        def calls(stream):
            for _ in range(20):
                K.ssm_scan_fwd(x, x, A, B, B, stream=stream)

        streams = [torch.cuda.Stream(), torch.cuda.Stream()]
        threads = [threading.Thread(target=calls, args=(streams[i % 2],)) for i in range(4)]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        worst = [ctypes.c_int.in_dll(counts, n).value for n in ("worst_on_a_stream", "worst_in_all")]
        print(f"at once: {worst[0]} on a stream, {worst[1]} in all", flush=True)
    return 0


if __name__ == "__main__":
    sys.exit(main())
