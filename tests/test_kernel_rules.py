"""Rules of ordering that the kernels keep, checked in their sources: breaking one is a race, which a run need not show (no GPU needed)."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2508_15919_b200", "csrc")


def _source(name):
    return re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())


def _between(src, start, end):
    i = src.index(start)
    return src[i:src.index(end, i)]


def test_simulator_orders_an_admission_before_its_commit():
    # single lanes note what is admitted (s_park, s_word, s_byte); the commit reads the notes with other lanes
    src = _source("hfx_sim.cu")
    last_note = src.rindex("park(adm_cnt", 0, src.index("parked(e0"))
    between = src[last_note:src.index("parked(e0")]
    # in a block that every iteration with an admission passes (not inside `if (from_list)` or a loop over the list)
    assert re.search(r"if \(adm_cnt > 0\) __syncwarp\(\);", between)


def test_simulator_orders_reading_a_slot_before_the_samples_overwrite_it():
    # the TTFT samples are closed up over the slots of the same 32 rows, of which those in flight are read just before
    src = _source("hfx_sim.cu")
    assert "__syncwarp();" in _between(src, "s_slot[i] >> 32);\n            last", "s_slot[n_ttft")


def test_simulator_orders_reading_a_finished_slot_before_an_admission_writes_it():
    # the lane that holds a slot reads its notes when its request finishes; the lane that holds an admitted request writes them
    src = _source("hfx_sim.cu")
    last_read, first_write = src.rindex("s_rctx[32 * k + lane]"), src.index("s_rinfo[32 * k + to] =")
    assert last_read < first_write and src.rindex("s_rinfo[32 * k + lane]") < last_read
    between = src[last_read:first_write]
    loop_end = between.index("nf = r_fin[k]")
    # behind the loop over the slots, in front of the list, so that an empty list does not leave it out
    assert "__syncwarp();" in between[loop_end:between.index("for (int s0 = 0; s0 < n_list")]


def test_dispatch_walk_reads_the_cursor_before_the_walking_warp_moves_it():
    # the first warp walks while the others look up and stage; what it writes for the next round must not reach a warp that is late with reading
    src = _source("hfx_dispatch.cu")
    body = _between(src, "for (;;) {\n    __syncthreads();\n    const int k_now = s_k;", "s_cursor = jumped;")
    read = body.index("cursor = s_cursor;")
    assert read < body.index("__syncthreads();", read) < body.index("break;", read)      # (every thread passes it)


def test_block_prefix_keeps_its_words_until_the_next_barrier():
    # what block_prefix returns is read from its shared array by every lane; one lane of the warp must not write there before a barrier
    src = _source("hfx_dispatch.cu")
    for m in re.finditer(r"block_prefix2?(?:<\w+>)?\([^;]*\b(s_part(?:64)?)\b[^;]*;", src):
        if m.group().startswith("block_prefix2(int64_t &x"):
            continue
        behind = src[m.end():]
        behind = behind[:min(behind.index("__syncthreads();"), behind.index("block_prefix") if "block_prefix" in behind else len(behind))]
        assert not re.search(m.group(1) + r"\[[^\]]*\] =[^=]", behind), behind


def _functions(src, word):
    """(header, body) of every function definition that is introduced by `word`."""
    out = []
    for m in re.finditer(word, src):
        brace = re.compile(r"[{;]").search(src, m.end())      # (a declaration ends without a body)
        if brace is None or brace.group() == ";":
            continue
        depth, i = 1, brace.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(src[i], 0)
            i += 1
        out.append((src[m.start():brace.start()], src[brace.end():i]))
    return out


def test_kernels_set_up_beside_the_one_in_front_read_nothing_through_the_read_only_path():
    # That path is for data that nothing writes while the kernel lives, and such a kernel lives while the one in front still writes.
    seen = set()
    for name in sorted(os.listdir(CSRC)):
        src = _source(name)
        kernels = _functions(src, r"__global__")
        early = [(h, b) for h, b in kernels if "cudaGridDependencySynchronize" in b]
        helpers = _functions(src, r"__device__") if kernels and len(early) == len(kernels) else []      # (a file of such kernels alone: its helpers too)
        for head, body in early + helpers:
            assert "__ldg(" not in body and "ld.global.nc" not in body and not re.search(r"const \w+ \*\s*__restrict__", head), (name, head)
        seen |= {re.search(r"\b(k_\w+)\s*\(", h).group(1) for h, _ in early}
    assert {"k_front", "k_replicas", "k_pd_rows", "k_pd_clock", "k_slo_assign", "k_disp_chain", "k_disp_assign"} <= seen


def test_kernels_behind_the_grid_barrier_ask_whether_it_was_given_up():
    # a barrier that ran out leaves the tiles, the running totals and the order unwritten: walking them reads and writes out of range
    kernels = {re.search(r"\b(k_\w+)\s*\(", h).group(1): b for h, b in _functions(_source("hfx_dispatch.cu"), r"__global__")}
    assert "grid_barrier(" in kernels["k_disp_sort"]
    for name, first_use in (("k_disp_chain", "tile_sum"), ("k_disp_assign", "run_end")):
        asked = kernels[name].index("CTL_ABORT")
        assert kernels[name].index("cudaGridDependencySynchronize") < asked < kernels[name].index(first_use), name


def test_what_is_kept_for_the_next_call_follows_what_was_launched():
    # a copy is changed for the other one behind the launch of the kernel that uses it and clears the other
    step, slo, disp, pd = (_source(f) for f in ("hfx_step.cu", "hfx_slomap.cu", "hfx_dispatch.cu", "hfx_pd.cu"))
    assert re.search(r"if \(rc == HFX_OK\) \{[^}]*tot_parity \^= 1u;\s*\}", step)
    assert slo.index("cudaLaunchKernelEx(&cfg, k_slo_window") < slo.index("slo_parity ^= 1u")
    # counters that the last kernel of a call clears: cleared by the next call where that kernel was not launched
    for src, last in ((disp, "cudaLaunchKernelEx(&cfg, k_disp_assign"), (pd, "cudaLaunchKernelEx(&cfg, k_pd_clock")):
        assert src.index("unsettled = true;") < src.index(last) < src.index("unsettled = false;")
        assert re.search(r"if \([\w>-]*unsettled\b[^;]*cudaMemsetAsync", src)


def test_every_refused_runtime_call_has_its_error_read():
    # an error left behind is what the next call's check finds (the caller of the *_configure functions reads theirs)
    for name in sorted(os.listdir(CSRC)):
        src = _source(name)
        configure = [b for h, b in _functions(src, r"int hfx_\w+_configure\(\)")]
        for m in re.finditer(r"return [^;]*HFX_E_CUDA;", src):
            if not any(m.group() in b for b in configure if "cudaFuncSetAttribute" in b and b in src and src.index(b) < m.start() < src.index(b) + len(b)):
                assert "cudaGetLastError()" in src[max(0, m.start() - 60):m.end()], (name, src[m.start() - 100:m.end()])
