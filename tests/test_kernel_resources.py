"""Registers and spills of the small kernels that a pass runs between its projections and of the sublayers that hold their weights in registers, as the
compiler reports them, and sizes of prefetches.

The small ones are bound by one memory round trip each, and the registers they hold are kept from the projection behind them.  The sublayers' kernels sit close to
the most that a thread can have."""
import os
import re
import subprocess

import pytest

from paper_2205_10350_b200 import build

NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
pytestmark = pytest.mark.skipif(not os.path.exists(NVCC), reason="no CUDA compiler")


def _report(tmp_path, kernels):
    """{kernel's symbol: (registers, bytes spilled)} of the kernels named."""
    src = tmp_path / "kernels.cu"
    src.write_text("".join(f'#include "{h}.cuh"\n' for h in ("accept", "attention_few", "ffn_few", "sublayer_f32")) +
                   "using namespace ad;\nvoid* kernels[] = {%s};\n" % ", ".join(f"(void*){k}" for k in kernels))
    r = subprocess.run([NVCC, "-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-std=c++17", "-rdc=true", "-I", build.CSRC, "-Xptxas", "-v",
                        "-c", str(src), "-o", str(tmp_path / "kernels.o")], check=True, capture_output=True, text=True)
    found = re.findall(r"Compiling entry function '(\S+)'.*?(\d+) bytes spill stores.*?Used (\d+) registers", r.stdout + r.stderr, re.S)
    names = {re.match(r"(?:\w+::)*(\w+)", k).group(1) for k in kernels}
    return {sym: (int(regs), int(spill)) for sym, spill, regs in found if any(re.match(rf"_ZN2ad\w*?\d+{n}(I|E)", sym) for n in names)}


def test_layernorm_holds_what_its_partial_sums_need(tmp_path):
    limits = {"layernorm_kernel": {4: 48, 8: 64, 16: 96}, "layernorm_many_kernel": {4: 64, 8: 64, 16: 112}}
    cases = [(n, t, p) for n in limits for t in (128, 256) for p in (4, 8, 16)]
    found = _report(tmp_path, [f"{n}<{a}, {t}, {p}>" for n, t, p in cases for a in ("bf16", "float")])
    assert len(found) == 2 * len(cases)
    for sym, (regs, spill) in found.items():
        name, p = re.search(r"(layernorm\w*kernel)I.*?Li\d+ELi(\d+)E", sym).groups()
        assert spill == 0 and regs <= limits[name][int(p)], f"{sym}: {regs} registers, {spill} bytes spilled"


def test_accept_kernels_fit_a_thousand_threads_without_spills(tmp_path):
    found = _report(tmp_path, [f"argmax_accept_kernel<{form}>" for form in ("ACC_ONE", "ACC_CLUSTERED", "ACC_ROWS")])
    assert len(found) == 3
    for sym, (regs, spill) in found.items():
        assert spill == 0 and regs <= 64, f"{sym}: {regs} registers, {spill} bytes spilled"


def test_sublayers_with_their_weights_in_registers_do_not_spill(tmp_path):
    few = [f"few::attention_few_kernel<{q}, {split}, {first}, {loop}>" for q in ("false", "true") for split in (1, 2) for first in ("false", "true")
           for loop in ("false", "true")] + ["few::ffn_few_kernel"]
    f32 = [f"sub32::sublayer_f32_kernel<sub32::{kind}, {d}, {s}, {loop}>" for kind, loop in (("SELF", "false"), ("CROSS", "false"), ("FFN", "false"), ("FFN", "true")) for d in (128, 256) for s in (32, 64)]
    parts = [f"layernorm_parts_kernel<{a}>" for a in ("bf16", "float")]
    found = _report(tmp_path, few + f32 + parts)
    assert len(found) == len(few) + len(f32) + len(parts)
    for sym, (regs, spill) in found.items():
        limit = 128 if "layernorm" in sym else 255             # (two CTAs of 256 threads an SM; the most a thread can have)
        assert spill == 0 and regs <= limit, f"{sym}: {regs} registers, {spill} bytes spilled"


def test_prefetches_end(tmp_path):
    """The pieces of a prefetch are counted in 32 bits: the step beyond the last one must not wrap around, for every number of CTAs."""
    src = tmp_path / "prefetch.cu"
    src.write_text("""
#include "ad_common.cuh"
using namespace ad;
int main() {
  const size_t sizes[] = {0, 16, 2048u * 1024, 5u << 21, PF_MAX, PF_MAX + 16, (size_t)1 << 31, ((size_t)1 << 32) - 16, (size_t)1 << 33};
  for (size_t s : sizes)
    for (uint32_t n = 1; n <= 1024; ++n) {
      const uint32_t b = prefetch_bytes(s);
      if (b > s || (uint64_t)b + (uint64_t)n * PF_PIECE > 0xffffffffull || b % 16) return 1;
    }
  return prefetch_bytes(PF_MAX) == PF_MAX && prefetch_bytes(((size_t)1 << 32) + 64) == 0 ? 0 : 1;
}
""")
    exe = tmp_path / "prefetch"
    subprocess.run([NVCC, "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-I", build.CSRC, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)]).returncode == 0
