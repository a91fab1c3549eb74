"""Registers and shared memory of the searches a handle takes by default, read from
ptxas (-Xptxas -v) for sm_103a: the blocks per SM that their launch bounds ask for
must fit, and no kernel may spill more than a few words.  A change that
breaks this costs speed without failing any result check."""
import os
import shutil
import subprocess
from concurrent.futures import ThreadPoolExecutor

import pytest

from test_build_resources import BLOCK_RESERVED_BYTES, CSRC, SM_REGISTERS, SM_SHARED_BYTES, _entry_resources

# mangled part, threads per block, blocks per SM, spilled bytes allowed
KERNELS = {
    "kmc_f32.cu": [("filter_search_kernelIfLi%dELb0ELi1EE", 32, 32, 16), ("filter_search_kernelIfLi%dELb0ELi4EE", 128, 8, 32),
                   ("filter_search_kernelIfLi%dELb0ELi8EE", 256, 4, 32), ("filter_search_kernelIfLi%dELb1ELi1EE", 32, 24, 80),
                   ("pairs_search_kernelILi%dELb0EE", 32, 32, 64), ("pairs_search_kernelILi%dELb1EE", 32, 32, 64),
                   ("search_kernelIfLi%dEEEv", 64, 16, 16)],
    "kmc_f64.cu": [("filter_search_kernelIdLi%dELb1ELi1EE", 32, 16, 48), ("filter_search_kernelIdLi%dELb1ELi8EE", 256, 2, 64),
                   ("search_kernelIdLi%dEEEv", 64, 8, 16)],
}


@pytest.fixture(scope="module")
def ptxas(tmp_path_factory):
    nvcc = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    if not os.path.exists(nvcc):
        nvcc = shutil.which("nvcc")
    if not nvcc:
        pytest.skip("nvcc not available")
    d = tmp_path_factory.mktemp("ptxas")

    def compiled(src):
        r = subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "-c",
                            os.path.join(CSRC, src), "-o", str(d / (src + ".o")), "-Xptxas", "-v"], capture_output=True, text=True)
        assert r.returncode == 0, r.stderr[-2000:]
        return r.stdout + r.stderr
    with ThreadPoolExecutor() as ex:
        return dict(zip(KERNELS, ex.map(compiled, KERNELS)))


@pytest.mark.parametrize("src,entry,threads,blocks,spill", [(s, *k) for s, ks in KERNELS.items() for k in ks],
                         ids=lambda v: v if isinstance(v, str) and "kernel" in v else "")
def test_default_searches_fit_their_blocks_per_sm(ptxas, src, entry, threads, blocks, spill):
    for dim in (2, 3):
        part = entry % dim
        log = ptxas[src]
        if part.startswith("search_kernel"):   # not filter_search_kernel or pairs_search_kernel
            part = "_ZN3kmc13" + part
        regs, smem, spilled = _entry_resources(log, part)
        per_warp = -(-regs // 8) * 8 * 32   # registers are given out by 256 per warp
        assert blocks * (threads // 32) * per_warp <= SM_REGISTERS, (part, regs)
        assert blocks * (smem + BLOCK_RESERVED_BYTES) <= SM_SHARED_BYTES, (part, smem)
        assert spilled <= spill, (part, spilled)
