"""CPU-side check of the bounded waits: all lanes of a warp get one answer.

A phase may complete between the last polls of two lanes.  Were a lane answered by its own polls alone, some lanes of the warp would
leave and the others go on into the next warp-wide instruction (a tcgen05.ld, a __syncwarp) without them.  The wait functions are taken
from the kernels' sources and compiled for the host, a thread per lane, with polls that succeed on some lanes and never on the others."""
import os
import re
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2512_03383_b200", "csrc")
USERS = {"tc.cuh": ["prefill.cu", "single.cu", "batch.cu"]}

HOST = r"""
#include <barrier>
#include <cstdint>
#include <cstdio>
#include <thread>
#include <vector>
#define __device__
static thread_local int lane;
static uint32_t answers;                                  // bit l: the polls of lane l succeed
static std::barrier<> meet(32);
static volatile bool votes[32];
static bool __all_sync(unsigned, bool v) {
  votes[lane] = v;
  meet.arrive_and_wait();
  bool all = true;
  for (int l = 0; l < 32; ++l) all = all && votes[l];
  meet.arrive_and_wait();
  return all;
}
static void __nanosleep(unsigned) {}
constexpr int %(limit)s = 200;
%(tries)s
%(waits)s
int main() {
  const uint32_t cases[] = {0xffffffffu, 0u, ~(1u << 7), 1u << 7, ~1u, 0x7fffffffu};
  for (uint32_t a : cases) {
    answers = a;
    volatile int flag = 0;
    uint32_t got = 0;
    bool r[32];
    std::vector<std::thread> t;
    for (int l = 0; l < 32; ++l) t.emplace_back([&, l] { lane = l; r[l] = %(call)s(0u, 0u, &flag); });
    for (auto& x : t) x.join();
    for (int l = 0; l < 32; ++l) got |= (uint32_t)r[l] << l;
    std::printf("%%08x %%08x %%d\n", a, got, flag);
  }
}
"""


def source(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def functions(text):
    """Name -> text of the device functions that poll or wait on an mbarrier."""
    out = {}
    for m in re.finditer(r"__device__ inline bool (p?mbar_(?:try|wait|poll)\w*)\([^)]*\) \{", text):
        depth, i = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(text[i], 0)
            i += 1
        out[m.group(1)] = text[m.start():i]
    return out


def calls(text, names):
    """(name, position) of every call outside the functions' own definitions."""
    for body in functions(text).values():
        text = text.replace(body, " " * len(body))
    return [(m.group(1), m.start(), text) for m in re.finditer(r"\b(%s)\(" % "|".join(names), text)]


def blocks_around(text, at):
    """The lines that open the blocks around a position."""
    depth, out = 0, []
    for i in range(at, -1, -1):
        if text[i] == "}":
            depth += 1
        elif text[i] == "{":
            if depth == 0:
                out.append(text[text.rfind("\n", 0, i) + 1:i])
            depth = max(0, depth - 1)
    return out


@pytest.mark.parametrize("where", sorted(USERS))
def test_all_lanes_of_a_warp_get_one_answer(where, tmp_path):
    funcs = functions(source(where))
    tries = [n for n in funcs if "_try" in n]
    used = {n for user in USERS[where] for n, _, _ in calls(source(user), funcs)}
    waits = sorted(n for n in used - set(tries) if not n.endswith("_lane"))
    assert waits
    for name in waits:
        prog = HOST % {
            "limit": "kPWait" if "kPWait" in "".join(funcs.values()) else "kWaitLimit",
            "tries": "\n".join("static bool %s(uint32_t, uint32_t) { return (answers >> lane) & 1; }" % n for n in tries),
            "waits": "\n".join(b for n, b in funcs.items() if n not in tries), "call": name}
        src, exe = tmp_path / (name + ".cpp"), tmp_path / name
        src.write_text(prog)
        subprocess.run(["g++", "-std=c++20", "-O1", "-pthread", str(src), "-o", str(exe)], check=True, timeout=120)
        lines = subprocess.run([str(exe)], check=True, capture_output=True, text=True, timeout=60).stdout.split("\n")[:-1]
        assert len(lines) == 6
        for polls, got, flag in (x.split() for x in lines):
            assert got == ("ffffffff" if polls == "ffffffff" else "00000000"), "%s: polls %s, answers %s" % (name, polls, got)
            assert flag == ("0" if polls == "ffffffff" else "1"), name


@pytest.mark.parametrize("user", sorted(sum(USERS.values(), [])))
def test_waits_of_one_lane_stand_in_code_of_one_lane(user):
    where = next(w for w, u in USERS.items() if user in u)
    for name, at, text in calls(source(user), functions(source(where))):
        line = text[text.rfind("\n", 0, at) + 1:text.find("\n", at)]
        if name.endswith("_lane"):
            assert any("lane == 0" in b for b in blocks_around(text, at)), line
        elif "_try" in name:                   # a poll of a lane decides nothing but how long the lane polls
            assert line.strip().startswith("for (") and line.rstrip().endswith("{}"), line


def test_lanes_of_the_decode_kernel_leave_with_the_status():
    """Its lanes keep their own answers and leave the kernel on their own: each that does writes the status (were it lane 0 alone,
    another lane could leave, the sums be wrong and the launch report none)."""
    text = source("decode.cu")
    assert not re.search(r"lane == 0\)\s*atomicExch\(c\.status", text)
    assert len(re.findall(r"auto give_up = \[&\]\(\) \{ atomicExch\(c\.status, UNIQL_ERR_TIMEOUT\); \};", text)) == 2
    waits = calls(text, ["mbar_wait"])
    assert len(waits) >= 7
    for _, at, rest in waits:
        behind = rest[at:at + 400]
        if re.search(r"\bok = $", rest[:at]):      # the producer, and the barrier of the consumers
            assert re.search(r"if \(!ok\) (break|give_up\(\))", behind), behind
        else:
            assert re.search(r"^[^;{]*\{\s*give_up\(\);\s*return;", behind), behind
    producer = text[text.index("if (!ok) {\n"):]
    assert re.search(r"\n\s*atomicExch\(c\.status, UNIQL_ERR_TIMEOUT\);\n\s*\}\n\s*return;", producer)
