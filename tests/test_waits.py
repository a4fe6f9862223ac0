"""Bounded waits of the tensor-core kernels: a warp that goes on to warp-wide (.aligned)
instructions gives up as a whole or not at all."""
import ctypes
import os
import re
import subprocess
import sys

import pytest
import torch

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1605_01715_gb300", "csrc")
# a use of TMEM by a role of the kernels, and what makes a wait's outcome the warp's before it
TMEM_USE = re.compile(r"\b(?:fold_acc<\w+>|tmem_ld8?(?:<\w+>)?|tmem_st32)\(")
WAIT = re.compile(r"\bmbar_wait(?:_ab|_warp)?\(")
VOTE = re.compile(r"__all_sync\(|bar_named_or\(")


@pytest.mark.parametrize("name,kernel", [("pair_tc.cuh", "void pair_tc_body("), ("sliced.cu", "k_sliced(")])
def test_every_tmem_use_follows_a_vote(name, kernel):
    text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
    body = text[text.index(kernel):]
    uses = list(TMEM_USE.finditer(body))
    assert uses
    for use in uses:
        last = list(WAIT.finditer(body, 0, use.start()))[-1]
        voted = last.group() == "mbar_wait_warp(" or VOTE.search(body, last.end(), use.start())
        assert voted, "%s: %s after a wait of single lanes: %s" % (name, use.group(), body[last.start():last.start() + 80])


@pytest.mark.gpu
@pytest.mark.parametrize("parity,raised,want", [
    ([1] * 32, 0, 1),                   # the barrier's phase is over: all pass
    ([1] * 32, 1, 1),                   # the same with the flag raised: complete comes first
    ([1] * 31 + [0], 1, 0),             # one lane gives up: all do
    ([0, 1] * 16, 1, 0),
    ([0] * 32, 1, 0),
])
def test_a_warp_gives_up_as_a_whole(parity, raised, want):
    import device_probe
    par = torch.tensor(parity, dtype=torch.int32, device="cuda")
    got = torch.full((32,), -1, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    assert device_probe.lib().probe_wait_warp(ctypes.c_void_p(par.data_ptr()), raised, ctypes.c_void_p(got.data_ptr())) == 0
    assert got.tolist() == [want] * 32


# A stand-in for the evaluation rows' launch: its wait gave up, and nothing was written.
FAKE = """
#include "%s/sliced.cuh"
namespace kifmm {
template <>
int launch_sliced_store<float>(const SlicedTable&, int, const int4*, int, const int*, const int*, const __half*,
                               const int*, const double*, float*, int, int* err, cudaStream_t s) {
    return cudaMemsetAsync(err, 1, 1, s) == cudaSuccess ? KIFMM_OK : KIFMM_ERR_CUDA;
}
}
"""

CHILD = """
import ctypes, sys
ctypes.CDLL(sys.argv[1], ctypes.RTLD_GLOBAL)      # before the library, so that its call comes here
import torch
from paper_1605_01715_gb300 import KifmmError, Plan, Tree
tree = Tree(torch.rand(3, 500, dtype=torch.float64, device="cuda"), max_leaf=32)
try:
    Plan(tree, kernel="sl", p=4, precision="mixed")
    print("plan made")
except KifmmError as e:
    print(e.status)
"""


@pytest.mark.gpu
def test_setup_reports_a_wait_that_gave_up(tmp_path):
    from paper_1605_01715_gb300 import build as kb
    src, so = tmp_path / "fake.cu", tmp_path / "fake.so"
    src.write_text(FAKE % CSRC)
    subprocess.run([kb.NVCC, "-shared", *kb.FLAGS, "-o", str(so), str(src)], check=True)
    r = subprocess.run([sys.executable, "-c", CHILD, str(so)], capture_output=True, text=True, cwd=os.path.dirname(kb.HERE),
                       timeout=300)
    assert r.stdout.strip() == "TIMEOUT", r.stdout + r.stderr
