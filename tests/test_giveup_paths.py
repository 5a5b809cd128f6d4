"""The give-up paths that no input reaches, checked on the source.

Stage 3 of the selector gives up (with an error status) when its phases run
past their limit or a bounded wait runs out. The block must leave its loop as
one: threads that go on would wait at barriers for those that left, and the
helper CTAs with them.

The few-rows linear gives up when a wait of any of its warps runs out: its TMA
loads in flight are then waited for, and a TMEM store before TMEM is released."""
import os
import re

from paper_2609_34867_gb300 import build as B


def test_every_thread_leaves_at_the_same_phase():
    code = open(os.path.join(B.CSRC, "p4q_diverse.cu")).read()
    code = re.sub(r"//[^\n]*", "", code)
    kernel = code[code.index("select_diverse_kernel(const DivArgs a)"):code.index("constexpr size_t kDivSmem")]
    loop = kernel[kernel.index("phase_limit = "):kernel.index("block_take_top")]
    # the exits: behind the loop's first barrier, on s.t, the waits' abort flag and the thread's own phase count
    exits = loop[loop.index("__syncthreads();"):]
    assert re.match(r"__syncthreads\(\);\s*const int t = s\.t;\s*if \(t >= a\.Kd \|\| s\.abort_flag\) break;\s*"
                    r"if \(phase >= phase_limit\) \{", exits)
    assert "for (int phase = 0;; ++phase)" in loop
    # no thread raises the flag by itself: only the bounded waits do, and those lie behind another barrier of the phase
    assert not re.search(r"abort_flag\s*=[^=]", kernel[kernel.index("phase_limit = "):])


def test_few_rows_leaves_nothing_in_flight():
    code = open(os.path.join(B.CSRC, "p4q_fewrows.cu")).read()
    code = re.sub(r"//[^\n]*", "", code)
    # the loads are waited for behind the barriers that every warp's abort precedes, not in the loading warp's own branch
    tail = code[code.rindex("else __syncthreads();"):]
    assert re.search(r"if \(threadIdx\.x == 0 && \*abort_flag\) \{[^}]*mbar_wait\(&full\[", tail)
    # the unpack loop may be left between a TMEM store and its wait: waited for behind it
    loop_end = code[code.index("tmem_st_16x256b_x8(ta"):]
    assert re.search(r"if \(ok\) ok = mbar_wait_all\(&acc_full[^;]*;\s*else tmem_st_wait\(\);", loop_end)
