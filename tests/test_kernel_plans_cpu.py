"""Host-side rules that kernels rely on, from the headers that hold them: compiled into a small host program."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2408_15766_b200", "csrc")


def run_host_program(tmp_path, header: str, body: str) -> str:
    src = tmp_path / "plan.cu"
    src.write_text(f'#include "{os.path.join(CSRC, header)}"\n#include <cstdio>\nusing namespace hass;\n{body}')
    exe = str(tmp_path / "plan")
    subprocess.run([os.environ.get("NVCC", "nvcc"), "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-o", exe, str(src)],
                   check=True)
    return subprocess.run([exe], capture_output=True, text=True).stdout


def test_blocks_that_add_up_groups_have_the_room_for_it(tmp_path):
    """A Normed Top-K block whose part of the columns leaves threads for several groups of tokens adds the groups' sums up in dynamic shared
    memory: for every part of every split the launch must have allocated it."""
    out = run_host_program(tmp_path, "normed_kernel.cuh", r"""
int main() {
    long long groups = 0, none = 0;
    for (int sms : {132, 148, 160})
        for (int d = 8; d <= 16384; d += 8)
            for (int K : {FIN_GRP, FIN_GRP + 1})
                for (int N = 1; N <= 260; ++N) {
                    const int split = normed_split(N, d, K, sms), bytes = normed_smem(d, split);
                    for (int rank = 0; rank < split; ++rank) {
                        const int units = part_begin(d / 8, rank + 1, split) - part_begin(d / 8, rank, split);
                        // as the kernel deals its threads out: `per` of them to a group
                        const int want = (units + 31) / 32 * 32, per = want < 32 ? 32 : want > NORMED_THREADS ? NORMED_THREADS : want;
                        if (NORMED_THREADS / per != gather_groups(units, NORMED_THREADS)) return std::printf("groups %d\n", units), 1;
                        if (NORMED_THREADS / per > 1) {
                            ++groups;
                            if (bytes < 8 * NORMED_THREADS * 4) return std::printf("room N %d d %d K %d split %d rank %d\n", N, d, K, split, rank), 1;
                        } else {
                            ++none;
                        }
                    }
                }
    std::printf("ok %d\n", groups > 0 && none > 0);
}
""")
    assert out == "ok 1\n", out


def test_handed_over_words_lie_where_their_reader_writes_next(tmp_path):
    """Eight epilogue warps: the first thread of a row may go on to its next tile while other rows' words are still being read. So no warp but
    the reader's own writes there: neither its staging buffers nor its columns of the pending logits hold another row's words."""
    out = run_host_program(tmp_path, "kernels.cuh", r"""
int main() {
    for (int thread = 64; thread < 192; ++thread) {
        const int quad = thread / 32 % 4;      // as the kernel has it
        for (int e = 0; e < 2; ++e) {          // a spill: two words
            const int at = meet_word(false, thread, e);
            if (at != meet_word(false, thread + 128, e)) return std::printf("two places, thread %d\n", thread), 1;
            if (at < stage_at(0, quad) || at + 4 > stage_at(0, quad) + SPILL_STAGES * SPILL_STAGE_BYTES)
                return std::printf("another warp's buffer, thread %d\n", thread), 1;
            for (int other = 64; other < 192; ++other)
                for (int e2 = 0; e2 < 2; ++e2)
                    if ((other != thread || e2 != e) && at == meet_word(false, other, e2)) return std::printf("shared, threads %d %d\n", thread, other), 1;
        }
        for (int e = 0; e < 2 + 2 * K_REG; ++e) {      // a list: entry q of the pending logits is 256 words behind entry q - 1
            const int at = meet_word(true, thread, e);
            if (at != meet_word(true, thread + 128, e) || at % 1024 != pending_at(thread) || at + 4 > 8 * SPILL_STAGES * SPILL_STAGE_BYTES)
                return std::printf("column, thread %d\n", thread), 1;
        }
    }
    std::printf("ok\n");
}
""")
    assert out == "ok\n", out


def test_rows_of_a_shared_tile_go_to_ctas_of_the_cluster(tmp_path):
    out = run_host_program(tmp_path, "kernels.cuh", r"""
int main() {
    for (int C = 2; C <= 8; ++C)
        for (int rows = 1; rows <= BM; ++rows) {
            const int per = piece_rows(rows, C);
            for (int r = 0; r < BM; ++r) {
                const int rank = piece_rank(r, per, C);
                if (rank < 0 || rank >= C) return std::printf("no such CTA: row %d of %d, %d CTAs\n", r, rows, C), 1;
                if (r < rows && (rank * per + r % per != r || r % per >= per)) return std::printf("row %d of %d, %d CTAs\n", r, rows, C), 1;
            }
        }
    std::printf("ok\n");
}
""")
    assert out == "ok\n", out
