"""The CPython module of a step's calls, against a library that only waits.  The calls let other Python threads run while they
are in the library (a launch into a full queue, or a copy from pageable memory, may wait for as long as the stream does), and
refuse what ctypes refused."""
import importlib.util
import os
import shutil
import subprocess
import sysconfig
import threading
import time

import numpy as np
import pytest

from paper_2607_22595_b200 import _build

# what the module links to, every call taking 300 ms
LIBRARY = """
#include <unistd.h>
#include "mix.h"
int mix_apply(mix_ctx* c, void* h, int T, float* s, void* stream) { usleep(300000); return T; }
int mix_set_slot_map(mix_ctx* c, const int* m, int T, int dev, void* stream) { usleep(300000); return T; }
int mix_set_request_map(mix_ctx* c, const int* r, int T, const int* s, int n, int dev, void* stream) { usleep(300000); return T + n; }
"""


class Tensor:
    """As much of a tensor as the module looks at."""

    def __init__(self, dtype, n):
        self.dtype, self.is_cuda, self.n = dtype, True, n

    def is_contiguous(self):
        return True

    def data_ptr(self):
        return 4096

    def size(self, dim):
        return self.n

    def numel(self):
        return self.n


@pytest.fixture(scope="module")
def fastcall(tmp_path_factory):
    folder = str(tmp_path_factory.mktemp("fastcall"))
    gcc = shutil.which("gcc")
    include = ["-I", os.path.join(_build.ROOT, "include")]
    with open(os.path.join(folder, "slow.c"), "w") as f:
        f.write(LIBRARY)
    subprocess.check_call([gcc, "-shared", "-fPIC", *include, "-o", os.path.join(folder, "libslow.so"), os.path.join(folder, "slow.c")])
    module = os.path.join(folder, "_fastcall.so")
    subprocess.check_call([gcc, "-O2", "-shared", "-fPIC", "-I", sysconfig.get_paths()["include"], *include, "-o", module,
                           os.path.join(_build.CSRC, "fastcall.c"), "-L", folder, "-lslow", "-Wl,-rpath,$ORIGIN"])
    spec = importlib.util.spec_from_file_location("_fastcall", module)
    m = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(m)
    return m


@pytest.mark.parametrize("name", ["apply", "set_slot_map", "set_request_map"])
def test_other_threads_run_during_a_call(fastcall, name):
    import torch
    args = {"apply": (1, Tensor(torch.bfloat16, 7), None, None, 16), "set_slot_map": (1, Tensor(torch.int32, 7), None, 16),
            "set_request_map": (1, Tensor(torch.int32, 7), Tensor(torch.int32, 5), None, 16)}[name]
    ticks, stop = [], threading.Event()

    def other():
        while not stop.is_set():
            ticks.append(time.perf_counter())
            time.sleep(0.005)

    thread = threading.Thread(target=other)
    thread.start()
    try:
        start = time.perf_counter()
        rc = getattr(fastcall, name)(*args)
        end = time.perf_counter()
    finally:
        stop.set()
        thread.join()
    assert rc == (12 if name == "set_request_map" else 7)
    assert end - start >= 0.3
    # 60 ticks fit into the call; without the GIL's release there is at most one, at either end
    assert sum(start + 0.01 < t < end - 0.01 for t in ticks) >= 5


@pytest.mark.parametrize("T_live", [3.7, "3", [3]])
def test_a_live_count_is_a_whole_number(fastcall, T_live):
    import torch
    with pytest.raises(TypeError):
        fastcall.set_slot_map(1, Tensor(torch.int32, 7), T_live, 16)
    with pytest.raises(TypeError):
        fastcall.set_request_map(1, Tensor(torch.int32, 7), Tensor(torch.int32, 5), T_live, 16)
    assert fastcall.set_slot_map(1, Tensor(torch.int32, 7), np.int32(3), 16) == 3
