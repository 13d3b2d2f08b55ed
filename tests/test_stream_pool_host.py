"""CPU check of the server's stream sets: a set whose creation failed (no device is visible to the
child process, so the first CUDA call returns an error) is not kept for the next request, and an
incomplete set that is handed back is dropped."""
import os
import subprocess

from paper_2106_03872_gb300 import build

PROGRAM = r"""
#include <cstdio>
#include "engine.h"
using namespace ks;
// 1: the pool throws, as it must without a device; 0: it handed out a set
static int refused(DevicePool& pool) {
  try {
    pool.take_streams();
    return 0;
  } catch (const Error&) {
    return 1;
  }
}
int main() {
  DevicePool pool(1 << 20);
  int threw = 0;
  try {
    StreamHolder h;
    h.acquire(&pool);
  } catch (const Error&) {
    threw = 1;
  }
  const int after_failure = refused(pool);
  pool.give_streams(StreamSet{});
  const int after_empty = refused(pool);
  std::printf("%d %d %d\n", threw, after_failure, after_empty);
  return 0;
}
"""


def test_failed_stream_set_is_not_pooled(tmp_path):
    if not os.path.exists(build.LIB):
        build.build()
    src, exe = str(tmp_path / "pool.cu"), str(tmp_path / "pool")
    with open(src, "w") as f:
        f.write(PROGRAM)
    subprocess.run([build.nvcc()] + build.ARCH + build.FLAGS + ["-I" + build.CSRC, src, build.LIB, "-Xlinker",
                    "-rpath=" + os.path.dirname(build.LIB), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120,
                       env=dict(os.environ, CUDA_VISIBLE_DEVICES=""))
    assert r.returncode == 0, r.stderr
    assert r.stdout.split() == ["1", "1", "1"]
