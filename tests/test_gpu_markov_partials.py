"""The Markov pick's merge of the bias kernel's partials, launched by itself
with more partials than a GPU of 256 SMs writes: a thread of the pick then
merges two, and a mark of a NaN or +inf entry must survive that."""
import ctypes
import os
import subprocess

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCE = r"""
#include "markov.cu"
extern "C" int pick(int greedy, int B, int V, int r, int G, float tau, const void* U, const void* W1, const void* W2T,
                    const int64_t* requests, void* E, void* part, void* sub, int nsub_pad, uint32_t* req_bad,
                    int32_t* drafts, float* conf, int32_t* status) {
  using namespace spec;
  MarkovLaunch p{};
  p.U = static_cast<const __nv_bfloat16*>(U);
  p.W1 = static_cast<const __nv_bfloat16*>(W1);
  p.W2T = static_cast<const __nv_bfloat16*>(W2T);
  p.r = r;
  p.B = B;
  p.K = 1;
  p.V = V;
  p.c2 = (float)(1.4426950408889634 / (tau > 0.0f ? tau : 1.0f));
  p.inv_t = 1.0f;
  p.seeds = p.request_ids = reinterpret_cast<const uint64_t*>(requests);
  p.pos_base = requests;
  p.E = static_cast<__nv_bfloat16*>(E);
  p.part = static_cast<MkPartial*>(part);
  p.sub = static_cast<float2*>(sub);
  p.nsub = (V + kMkSub - 1) / kMkSub;
  p.nsub_pad = nsub_pad;
  p.G = G;
  p.req_bad = req_bad;
  p.drafts = drafts;
  p.conf = conf;
  p.status = status;
  if (greedy) markov_pick_kernel<true><<<B, kPickThreads>>>(p);
  else markov_pick_kernel<false><<<B, kPickThreads>>>(p);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    from paper_2607_25852_gb300 import build
    d = tmp_path_factory.mktemp("pick")
    src, out = d / "pick.cu", d / "pick.so"
    src.write_text(SOURCE)
    subprocess.run([build.NVCC, *build.ARCH, *build.FLAGS, "-I", build.CSRC, "-shared", str(src), "-o", str(out)],
                   check=True, capture_output=True)
    return ctypes.CDLL(str(out))


@pytest.mark.parametrize("greedy", [True, False])
@pytest.mark.parametrize("at", [(5, 5 + 1024), (1029, 5), (3, 700)])
def test_a_marked_partial_survives_the_merge(lib, greedy, at):
    """Partial at[0] is marked bad and holds no maximum, partial at[1] holds the
    row's; the others are empty.  Request 1 is the same without the mark."""
    dev, B, V, r, G = "cuda", 2, 512, 64, 300
    bf = lambda *s: torch.zeros(s, dtype=torch.bfloat16, device=dev)
    part = np.zeros((B, 4 * G), dtype=[("m", "f4"), ("s", "f4"), ("L", "f4"), ("idx", "i4"), ("M", "f4"),
                                       ("flags", "i4"), ("pad", "i4", 2)])
    assert part.itemsize == 32
    part["m"] = part["L"] = -np.inf
    part["idx"] = 2**31 - 1
    part["flags"][0, at[0]] = 1
    part["m"][:, at[1]], part["s"][:, at[1]], part["L"][:, at[1]], part["idx"][:, at[1]] = 1.0, 1.0, 1.0, 300
    part_d = torch.as_tensor(part.view(np.uint8).reshape(B, -1).copy(), device=dev)
    sub = torch.zeros((B, 16, 2), device=dev)  # 8 sub-blocks of 64 columns in use
    sub[:, :, 0] = float("-inf")
    sub[:, 4] = torch.tensor([1.0, 1.0], device=dev)
    U, W1, W2T, E = bf(B, 1, V), bf(V, r), bf(V, r), bf(128, r)
    U.fill_(-1e4)
    U[:, 0, 300] = 1.0
    i32 = lambda *s: torch.zeros(s, dtype=torch.int32, device=dev)
    req, bad, z, status = torch.full((B,), 7, dtype=torch.int64, device=dev), i32(B), i32(B, 1), i32(1)
    conf = torch.zeros((B, 1), device=dev)
    torch.cuda.synchronize()
    ptr = lambda t: ctypes.c_void_p(t.data_ptr())
    assert lib.pick(int(greedy), B, V, r, G, ctypes.c_float(0.0 if greedy else 1.0), ptr(U), ptr(W1), ptr(W2T),
                    ptr(req), ptr(E), ptr(part_d), ptr(sub), 16, ptr(bad), ptr(z), ptr(conf), ptr(status)) == 0
    assert z[:, 0].tolist() == [-1, 300]
    assert conf[0].item() == 0.0 and conf[1].item() > 0.99
    assert status.item() == 4  # SPEC_ERR_BAD_INPUT
