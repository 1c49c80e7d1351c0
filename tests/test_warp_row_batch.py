"""The packed rows of a warp's batch (RowBatch): a row is written only after a __syncwarp that follows every lane's reads of
the batch before, and read only after one that follows its write (shuffles and votes order no memory). On the host, with
the class's own text and rows that remember who touched them."""
import subprocess

import pytest

import warp_emu

DRIVER = r"""
struct Tracked {
    uint32_t x = 0, y = 0, z = 0, w = 0;
    Tracked() = default;
    Tracked(uint32_t a, uint32_t b, uint32_t c, uint32_t d) : x(a), y(b), z(c), w(d) {}
    Tracked(const Tracked& o) : x(o.x), y(o.y), z(o.z), w(o.w) { touch(&o, false); }
    Tracked& operator=(const Tracked& o) {
        x = o.x, y = o.y, z = o.z, w = o.w;
        touch(this, true);
        return *this;
    }
    static void touch(const Tracked* p, bool write);
};
static Tracked rows[32];
static int last[32][32][2];  // per row, lane and kind: __syncwarps that the lane had passed, and one
static bool raced;
void Tracked::touch(const Tracked* p, bool write) {
    if (p < rows || p >= rows + 32) return;
    const int lane = emu::cur->tid.x, at = (int)emu::cur->syncs + 1;
    for (int l = 0; l < 32; ++l)
        for (int k = 0; k < 2; ++k)
            if (l != lane && (write || k) && last[p - rows][l][k] >= at) raced = true;
    last[p - rows][lane][write] = at;
}
#define uint4 Tracked
static Tracked make_uint4(uint32_t a, uint32_t b, uint32_t c, uint32_t d) { return Tracked(a, b, c, d); }
struct SampleArgs {
    const uint32_t* tau;
    int rk;
};
struct SampleBlock {
    Tracked operator()(uint32_t q, int) const { return Tracked(q, q, q, q); }
};
static bool coin_live(uint32_t x, uint32_t t) { return x * 2654435761u < t; }
//KERNELS//
int main(int argc, char** argv) {
    const unsigned seed = atoi(argv[1]);
    uint64_t live = 0, want = 0;
    SampleArgs a{nullptr, 0};
    emu::run(32, 0, 1, seed, [&] {
        const uint32_t lane = threadIdx.x;
        for (uint32_t batch = 0; batch < 6; ++batch) {
            const uint32_t deg = (lane * 7 + batch * 5 + seed) % 23, lo = 1000 * batch + 31 * lane, tau = 1u << 30;
            for (uint32_t e = lo; e < lo + deg; ++e) want += coin_live(e >> 2, tau);
            const RowBatch rb(rows, lo, lo + deg, tau, row_quads(lo, lo + deg));
            uint32_t st = 0;
            for (uint32_t base = 0; base < rb.total; base += 64)
                rb.step(a, SampleBlock(), base, &st, [&](uint32_t, unsigned m) {
                    if (!__any_sync(kFull, m != 0)) return;
                    live += __popc(m);
                });
        }
    });
    fprintf(stderr, "live %llu of %llu, raced %d\n", (unsigned long long)live, (unsigned long long)want, raced);
    return live != want ? 1 : raced ? 2 : 0;
}
"""


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    return warp_emu.build(tmp_path_factory.mktemp("rows"), "sample.cu", ["quad_live", "row_quads", "RowBatch"], DRIVER)


@pytest.mark.parametrize("seed", range(8))
def test_rows_are_packed_after_the_last_batch_is_read(exe, seed):
    r = subprocess.run([exe, str(seed)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stderr
