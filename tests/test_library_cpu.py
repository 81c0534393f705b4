"""CPU-side checks of the product: the C-ABI library builds, loads and exports every symbol the
header declares; argument validation that needs no GPU; the binding fails loudly without it."""
import ctypes
import os
import re
import subprocess

import pytest

from paper_2605_08840_b200 import binding as rk
from paper_2605_08840_b200 import build as rk_build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def lib():
    rk_build.build()
    return rk.load_library()


def declared_symbols():
    text = open(os.path.join(ROOT, "include", "restkv.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(restkv_[a-z_]+)\s*\(", text)))


def test_header_and_binding_agree_on_the_exports():
    assert declared_symbols() == sorted(rk.EXPORTS)


def test_library_exports_every_declared_symbol(lib):
    for name in declared_symbols():
        assert hasattr(lib, name), name


def test_error_strings(lib):
    for code in range(6):
        assert rk.error_string(code) not in ("", "unknown status")
    assert rk.error_string(99) == "unknown status"


def test_workspace_bytes_validates_without_a_gpu(lib):
    ok = rk.make_shape(1, 32, 8, 128, 131072, 32)
    n = lib.restkv_workspace_bytes(ctypes.byref(ok), 2048)
    assert n > 0 and n % 256 == 0
    assert lib.restkv_workspace_bytes_adaptive(ctypes.byref(ok), 2048) > n
    for bad in (rk.make_shape(1, 7, 2, 128, 100, 32),          # heads not divisible
                rk.make_shape(1, 8, 2, 128, 100, 32, causal_tail=3),
                rk.make_shape(1, 8, 2, 128, 32, 32, causal_tail=32),   # no scored rows left
                rk.make_shape(0, 8, 2, 128, 100, 32),
                rk.make_shape(1, 8, 2, 20, 100, 32),
                rk.make_shape(1, 8, 2, 128, 100, 32, dtype=5)):
        assert lib.restkv_workspace_bytes(ctypes.byref(bad), 16) == 0
    assert lib.restkv_workspace_bytes(None, 16) == 0


def test_null_handle_is_rejected(lib):
    assert lib.restkv_destroy(None) == rk.ERR_INVALID_ARG
    assert lib.restkv_poll_status(None, None) == rk.ERR_INVALID_ARG
    assert lib.restkv_launch_count(None) == 0
    shape = rk.make_shape(1, 8, 2, 64, 100, 32)
    pool = rk.fixed_pool(7)
    assert lib.restkv_score(None, ctypes.byref(shape), None, None, None, 0.9, ctypes.byref(pool), None, None, None,
                            0, None) == rk.ERR_INVALID_ARG


def test_no_silent_fallback_when_the_library_is_missing(monkeypatch, tmp_path):
    monkeypatch.setattr(rk, "_lib", None)
    monkeypatch.setattr(rk, "LIB_PATH", str(tmp_path / "missing.so"))
    with pytest.raises(RuntimeError, match="no CPU fallback"):
        rk.load_library()


def test_product_does_not_import_the_oracle():
    pkg = os.path.join(ROOT, "paper_2605_08840_b200")
    for dirpath, _, files in os.walk(pkg):
        for f in files:
            if f.endswith((".py", ".cu", ".cuh", ".h")):
                src = open(os.path.join(dirpath, f)).read()
                assert "oracle" not in src.lower() or f == "inputs.py", f
    for f in os.listdir(os.path.join(ROOT, "oracle")):
        if f.endswith((".py", ".c")):
            src = open(os.path.join(ROOT, "oracle", f)).read()
            assert "paper_2605_08840_b200" not in src and "librestkv.so" not in src, f


def test_accumulator_phases_take_arrivals_of_their_own_tile_only():
    """Score kernel from given statistics: a stage's kv_empty and acc_full count three arrivals a tile, of the two warps that sum
    ||v||^2 and of the products' commit.  Every order in which the roles can run, with the warps' two arrivals in the order that the
    source has them: no arrival may count for another tile than its own."""
    source = open(os.path.join(ROOT, "paper_2605_08840_b200", "csrc", "tc_fused.cu")).read()
    body = source[source.index("void half_terms("):]
    order = re.findall(r"mbar_arrive\(&cx\.B->(\w+)\[", body[:body.index("\n}\n")])
    assert sorted(order) == ["acc_full", "kv_empty"]
    tiles = 3                                      # of one stage
    helper = [(t, bar) for t in range(tiles) for bar in order]
    commit = [(t, bar) for t in range(tiles) for bar in ("acc_full", "kv_empty")]
    seen, todo = set(), [(0, 0, 0)]                # operations that the two warps and the issuing thread have done
    while todo:
        state = todo.pop()
        if state in seen:
            continue
        seen.add(state)
        done = [op for ops, n in zip((helper, helper, commit), state) for op in ops[:n]]
        phase = {bar: sum(1 for _, b in done if b == bar) // 3 for bar in ("acc_full", "kv_empty")}
        for role, ops in enumerate((helper, helper, commit)):
            if state[role] == len(ops):
                continue
            tile, bar = ops[state[role]]
            # the stage holds the tile once kv_empty has let the loader refill it; the products also want the epilogue to have
            # read the accumulators of the tile before
            if phase["kv_empty"] < tile or (role == 2 and phase["acc_full"] < tile):
                continue
            assert phase[bar] == tile, "an arrival of tile %d counts for tile %d of %s" % (tile, phase[bar], bar)
            todo.append(tuple(n + (r == role) for r, n in enumerate(state)))
    assert (len(helper), len(helper), len(commit)) in seen


def test_index_sums_of_the_longest_rows(tmp_path):
    """The sum of the indices whose keys lie above a limit, at both ends of the indices
    that a row of up to 2^31 - 1 keys has, or one of up to 2^30."""
    source = tmp_path / "sums.cc"
    source.write_text("""
#include <cstdio>
#include <initializer_list>
#include "index_sum.cuh"
template <bool kShort>
void print(unsigned int i) {
  for (unsigned int m = 0; m < 16; ++m) {
    unsigned long long sum = 5;
    restkv::add_indices_above<kShort>(sum, i, 7 + (m & 1), 7 + (m >> 1 & 1), 7 + (m >> 2 & 1), 7 + (m >> 3), 7);
    std::printf("%u %u %llu\\n", i, m, sum);
  }
}
int main() {
  for (unsigned int i : {0u, 1u, (1u << 30) - 4u}) print<true>(i);
  for (unsigned int i : {0u, 1u, (1u << 30) - 4u, (1u << 30) - 1u, 1u << 30, 0x7FFFFFF8u, 0x7FFFFFFBu}) print<false>(i);
}
""")
    program = tmp_path / "sums"
    subprocess.run(["g++", "-std=c++17", "-I", rk_build.CSRC, "-o", str(program), str(source)], check=True)
    lines = subprocess.run([str(program)], check=True, capture_output=True, text=True).stdout.split("\n")[:-1]
    assert len(lines) == 10 * 16
    for line in lines:
        i, m, total = (int(x) for x in line.split())
        assert total == 5 + sum(i + k for k in range(4) if m >> k & 1), line
