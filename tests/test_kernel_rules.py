"""Rules of the machine that the GEMM kernel has to keep where no result shows it: checked on its source."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2507_19131_b200", "csrc")


def kernel_source():
    """csrc/gemm_tc.cu's k_gemm_tc without comments."""
    text = open(os.path.join(CSRC, "gemm_tc.cu")).read()
    body = text[text.index("k_gemm_tc(const"):text.index("// ---- host side")]
    return re.sub(r"//[^\n]*", "", body)


def test_the_lane_that_issued_the_mmas_commits_them_when_the_cta_gives_up():
    """tcgen05.commit covers what the executing thread has issued.  The MMAs are issued by the lane that elect.sync names (the
    same one for a full warp every time), so the commit in front of freeing tensor memory has to be that lane's too."""
    body = kernel_source()
    give_up = body[body.index("if (*abort_flag) {"):]
    assert re.search(r"if \(warp == 1 && elect_one\(\)\) mma_commit\(bar_drain\);", give_up)
    assert len(re.findall(r"mma_commit\(bar_drain\)", body)) == 1
    issuer = body[body.index("} else if (warp == 1) {"):body.index("} else if (warp < FIRST_UNPACK_WARP)")]
    assert "const bool leader = elect_one();" in issuer and re.search(r"if \(leader\) \{[^}]*mma_i8\(", issuer)


def test_registers_are_exchanged_by_whole_warpgroups():
    """setmaxnreg is executed by all warps of a warpgroup, the same instruction: one for the side warps in front of the split into
    roles, one for the epilogue warps, under conditions that are the same for every four warps."""
    text, body = open(os.path.join(CSRC, "gemm_tc.cu")).read(), kernel_source()
    assert len(re.findall("setmaxnreg", body)) == 2
    assert re.search(r'\n  if \(epi_regs\(EW, PACKED\) > 0 && warp < FIRST_EPI_WARP\) asm volatile\("setmaxnreg\.dec\.[^\n]*\n\s*'
                     r'if \(warp == 0\) \{', body)
    assert re.search(r'\n  \} else \{\s*if \(epi_regs\(EW, PACKED\) > 0\) asm volatile\("setmaxnreg\.inc\.', body)
    number = {n: int(v) for n, v in re.findall(r"\b(FIRST_UNPACK_WARP|UNPACK_WARPS|CODE_WARPS|F32_WARPS) = (\d+)", text)}
    assert len(number) == 4 and all(v % 4 == 0 for v in number.values())      # every boundary between roles lies between warpgroups


def test_the_lanes_of_a_warp_give_up_together():
    """A bounded wait that runs out in one lane only would leave the others at the next aligned instruction for good: warps that
    walk converged wait with one answer for all lanes."""
    assert not re.findall(r"\bmbar_wait(?:<\w+>)?\(", kernel_source())
    calib = open(os.path.join(CSRC, "calib.cu")).read()
    epilogue = calib[calib.index("double part[CG_EPI_COLS]"):calib.index("// a wait ran out")]
    assert not re.findall(r"\bmbar_wait(?:<\w+>)?\(", epilogue) and "mbar_wait_warp(acc_full" in epilogue
    wait = open(os.path.join(CSRC, "tc_ptx.cuh")).read()
    wait = wait[wait.index("bool mbar_wait_warp("):wait.index("void tma_load_2d")]
    assert len(re.findall(r"if \(.*return", wait)) == len(re.findall(r"__(?:all|any)_sync\(0xffffffffu", wait)) == 3


def test_tensor_memory_is_read_by_converged_warps():
    """tcgen05.ld and its wait are for all lanes of a warp at once.  Lanes whose row is not stored leave a pass of an epilogue's loop
    early, so there is a __syncwarp between that and the next read."""
    def source(name):
        return re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
    calib = source("calib.cu")
    assert len(re.findall(r"\btmem_ld\(", calib)) == 1
    loop = calib[calib.index("for (int g = 0; g < CG_EPI_COLS; g += 8) {"):]
    assert "continue;" in loop[:loop.index("observe_warp(")]
    assert re.match(r"[^{]*\{\s*int32_t S\[CAL_SLICES\]\[8\];\s*__syncwarp\(\);\s*#pragma unroll\s*for [^;]*;[^;]*;[^;]*tmem_ld\(", loop)
    gemm = source("gemm_epilogue.cuh")
    assert re.search(r"clamp_pack4<MODE != EPI_FC1>\([^;]*;\s*\}\s*if \(TAPS\) __syncwarp\(\);\s*\}", gemm)          # taps of a half
    assert re.search(r"rows_left\) store_codes8\([^;]*;\s*__syncwarp\(\);\s*\}\s*return true;", gemm)                 # code outputs
    assert re.search(r"if \(!dst_ptr\[i\]\) continue;", gemm) and re.search(r"fetch\(ch \+ RES_SLOTS\);\s*__syncwarp\(\);\s*\};", gemm)
