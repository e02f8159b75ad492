// The library's host code over the stand-in runtime: one scenario a run (its name is the argument).
#include <c2kv.h>

#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <numeric>

#include "fake_cudart.h"

namespace {

#define CHECK(cond, ...)                                                \
    do {                                                                \
        if (!(cond)) {                                                  \
            std::printf("%s:%d: %s: ", __FILE__, __LINE__, #cond);      \
            std::printf(__VA_ARGS__);                                   \
            std::printf("\n");                                          \
            std::exit(1);                                               \
        }                                                               \
    } while (0)

alignas(256) char buffer[256];          // every tensor: its address is checked, nothing is read

struct Shape {
    int dtype, hq, hkv, d, layers = 1;
};

struct Context {
    Shape s;
    c2kv_ctx* ctx = nullptr;
    explicit Context(Shape shape, int split = 0, int pairs = 0, int fuse = 0, int impl = 0) : s(shape) {
        c2kv_config cfg{};
        cfg.layers = s.layers;
        cfg.n_q_heads = s.hq;
        cfg.n_kv_heads = s.hkv;
        cfg.head_dim = s.d;
        cfg.rope_theta = 1e4;
        cfg.dtype = s.dtype;
        cfg.pool_slots = 65536;
        cfg.attn_impl = impl;
        cfg.attn_split = split;
        cfg.attn_pairs = pairs;
        cfg.fuse = fuse;
        const c2kv_status st = c2kv_create(&cfg, nullptr, &ctx);
        CHECK(st == C2KV_OK, "create: %s", c2kv_last_error(nullptr));
    }
    ~Context() { c2kv_destroy(ctx); }
    int chunk(int slots) {
        int32_t id = -1;
        CHECK(c2kv_compress_chunk(ctx, buffer, buffer, slots, 1, C2KV_MODE_STORED, &id) == C2KV_OK, "compress");
        return id;
    }
    // `batch` requests of one chunk each
    c2kv_cache* compose(int batch, int slots, int suffix) {
        std::vector<int32_t> ptr(batch + 1), ids(batch, chunk(slots));
        std::iota(ptr.begin(), ptr.end(), 0);
        c2kv_cache* cache = nullptr;
        CHECK(c2kv_compose(ctx, batch, ptr.data(), ids.data(), nullptr, suffix, &cache) == C2KV_OK, "compose: %s",
              c2kv_last_error(ctx));
        return cache;
    }
    c2kv_status attend(c2kv_cache* cache, int suffix) {
        return c2kv_attend(ctx, cache, -1, buffer, buffer, buffer, suffix, buffer, nullptr);
    }
    c2kv_status decode(c2kv_cache* cache, int batch) {
        std::vector<int32_t> steps(batch, 0);
        return c2kv_decode(ctx, cache, -1, buffer, buffer, buffer, steps.data(), buffer, nullptr);
    }
    c2kv_status extract(int tokens, int ratio) {
        return c2kv_extract_attention(ctx, 1, buffer, buffer, buffer, tokens, ratio, buffer, nullptr);
    }
    c2kv_status step(int chunks, int slots, int suffix, c2kv_cache** cache) {
        std::vector<int32_t> ids;
        for (int i = 0; i < chunks; ++i) ids.push_back(chunk(slots));
        const int32_t ptr[2] = {0, chunks};
        return c2kv_compose_attend(ctx, 1, ptr, ids.data(), nullptr, suffix, buffer, buffer, buffer, suffix, buffer,
                                   nullptr, cache);
    }
};

constexpr int kBf16 = C2KV_DTYPE_BF16, kF32 = C2KV_DTYPE_F32;

// The kernels whose warps trade registers (setmaxnreg) wait forever when the launch holds fewer than
// the split hands out, so none of them may be launched with a smaller compiled count.  One kernel a run
// (the library reads the counts once a process), under the calls that launch them.
void registers(const std::string& part) {
    fake::registers = [&](const std::string& name) { return name.find(part) != std::string::npos ? 64 : 168; };
    int refused = 0;
    auto call = [&](c2kv_status st) { refused += st == C2KV_ERR_CUDA; };
    c2kv_cache* cache = nullptr;
    for (int d : {128, 64}) {
        Context pairs({kBf16, 32, 8, d}, 1, 1);
        call(pairs.attend(pairs.compose(1, 1000, 300), 300));
        call(pairs.extract(600, 4));
    }
    Context step({kBf16, 32, 8, 128});
    call(step.step(4, 128, 32, &cache));
    Context forced({kBf16, 32, 8, 128}, 0, 0, C2KV_FUSE_ALWAYS);
    call(forced.step(4, 128, 200, &cache));
    call(step.decode(step.compose(1, 1000, 8), 1));
    Context groups({kBf16, 64, 8, 128});                  // eight queries a KV head, more units than SMs
    call(groups.decode(groups.compose(20, 400, 8), 20));
    CHECK(!fake::launched(part), "%s launched with too few registers", part.c_str());
    CHECK(refused > 0, "no call reaches %s", part.c_str());
}

// What a process sets up on its first device is set up again on its second: every kernel that needs more
// than 48 KB of dynamic shared memory launches there too, and the rules count that device's SMs.
void second_device() {
    fake::sms = [](int device) { return device == 0 ? 152 : 16; };
    for (fake::device = 0; fake::device < 2; ++fake::device) {
        auto ok = [](c2kv_ctx* ctx, c2kv_status st, const char* what) {
            CHECK(st == C2KV_OK, "device %d, %s: %s", fake::device, what, c2kv_last_error(ctx));
        };
        for (const Shape& s : {Shape{kF32, 4, 2, 64}, Shape{kF32, 16, 4, 128}, Shape{kBf16, 24, 8, 64},
                               Shape{kBf16, 24, 8, 128}, Shape{kBf16, 32, 8, 64}, Shape{kBf16, 32, 8, 128}}) {
            Context one(s);
            for (int batch : {1, 40}) {                              // one row tile or key split a CTA; many
                c2kv_cache* cache = one.compose(batch, 700, 100);
                ok(one.ctx, one.attend(cache, 3), "attend");
                ok(one.ctx, one.attend(cache, 100), "attend");
                if (s.hq / s.hkv != 3) ok(one.ctx, one.decode(cache, batch), "decode");
            }
            ok(one.ctx, one.extract(600, 4), "extract");
            if (s.dtype == kBf16 && s.hq == 32) {
                Context pairs(s, 1, 1);
                ok(pairs.ctx, pairs.attend(pairs.compose(1, 700, 100), 100), "attend, pairs");
                ok(pairs.ctx, pairs.extract(600, 4), "extract, pairs");
            }
        }
        Context groups({kBf16, 64, 8, 128});
        ok(groups.ctx, groups.decode(groups.compose(20, 400, 8), 20), "decode of groups of eight");
        for (int fuse : {C2KV_FUSE_AUTO, C2KV_FUSE_ALWAYS}) {
            c2kv_cache* cache = nullptr;
            Context step({kBf16, 32, 8, 128}, 0, 0, fuse);
            ok(step.ctx, step.step(4, 128, fuse == C2KV_FUSE_AUTO ? 32 : 200, &cache), "step");
        }
        // 64 query tiles: one an SM on the first device, more than the SMs on the second
        fake::launches.clear();
        Context tiles({kBf16, 32, 8, 128}, 1);
        ok(tiles.ctx, tiles.attend(tiles.compose(2, 300, 100), 100), "attend, 64 tiles");
        CHECK(fake::launched("attn_solo_kernelILb0ELi128ELb1E") == (fake::device == 0), "device %d", fake::device);
    }
}

// Scratch that only makes a call faster is done without when it cannot be had: the partials of automatic
// key-range splits,
void no_partials() {
    Context one({kBf16, 32, 8, 128}), forced({kBf16, 32, 8, 128}, 4);
    c2kv_cache* cache = one.compose(1, 8192, 64);
    c2kv_cache* cache4 = forced.compose(1, 8192, 64);
    CHECK(one.attend(cache, 64) == C2KV_OK, "attend");
    CHECK(fake::launched("attn_combine_kernel"), "the call is split when there is memory");
    fake::launches.clear();
    fake::alloc_fails = [](size_t bytes) { return bytes > 64 * 32 * 128 * 2; };          // the turned queries fit
    CHECK(one.attend(cache, 64) == C2KV_OK, "attend without partials: %s", c2kv_last_error(one.ctx));
    CHECK(fake::launched("attn_solo_kernel") && !fake::launched("attn_combine_kernel"), "one split");
    CHECK(forced.attend(cache4, 64) == C2KV_ERR_NOMEM, "splits that were asked for");
}

// and the turned queries of a step of ragged chunks, which is composed before it is attended.
void no_queries() {
    Context step({kBf16, 32, 8, 128, 32}), never({kBf16, 32, 8, 128, 32}, 0, 0, C2KV_FUSE_NEVER);
    c2kv_cache* cache = nullptr;
    CHECK(step.step(10, 125, 64, &cache) == C2KV_OK, "step");
    CHECK(!fake::launched("14attn_tc_kernelILb1"), "not fused when there is memory");
    fake::launches.clear();
    fake::alloc_fails = [](size_t bytes) { return bytes == (size_t)32 * 64 * 32 * 128 * 2; };
    CHECK(step.step(10, 125, 64, &cache) == C2KV_OK, "step without turned queries: %s", c2kv_last_error(step.ctx));
    CHECK(fake::launched("14attn_tc_kernelILb1ELb0"), "fused");
    CHECK(never.step(10, 125, 64, &cache) == C2KV_ERR_NOMEM, "never fused");
}

// Few rows of many units on the CUDA cores: four rows a CTA, whose warps share the keys; not the forms of 16
// and 64 rows, most of which would be empty.
void few_rows() {
    for (int d : {64, 128}) {
        Context one({kF32, 32, 8, d, 32});
        for (int slots : {8, 100, 300}) {
            c2kv_cache* cache = one.compose(10, slots, 4);
            fake::launches.clear();
            CHECK(one.attend(cache, 1) == C2KV_OK, "attend: %s", c2kv_last_error(one.ctx));
            CHECK(fake::launched("attn_simt_kernelIfLi" + std::to_string(d) + "ELi0E"), "d %d, %d slots", d, slots);
        }
    }
}

// bf16 heads of 64 channels: few rows over few keys stay on the CUDA cores, for both attend calls.
void short64() {
    Context one({kBf16, 32, 8, 64, 32}), split({kBf16, 32, 8, 64, 32}, 1);
    struct {
        int slots, n;
        bool tc;
    } const cases[] = {{8, 1, false}, {300, 1, false}, {900, 1, true}, {30, 8, true}, {100, 60, true}};
    for (const auto& k : cases) {
        c2kv_cache* cache = one.compose(10, k.slots, 64);
        for (int noalloc = 0; noalloc < 2; ++noalloc) {
            fake::launches.clear();
            const c2kv_status st = noalloc ? c2kv_attend_noalloc(one.ctx, cache, k.slots > 100 ? 0 : -1, buffer, buffer,
                                                                 buffer, k.n, buffer, nullptr)
                                           : one.attend(cache, k.n);
            if (st == C2KV_ERR_ARG && noalloc) continue;          // beyond its fixed scratch
            CHECK(st == C2KV_OK, "%s", c2kv_last_error(one.ctx));
            if (noalloc && k.slots > 100) continue;               // one layer: another count of query tiles
            CHECK(fake::launched("attn_solo_kernel") == k.tc && fake::launched("attn_simt_kernel") != k.tc,
                  "%d slots, %d tokens, noalloc %d", k.slots, k.n, noalloc);
        }
        fake::launches.clear();
        CHECK(split.attend(split.compose(10, k.slots, 64), k.n) == C2KV_OK, "%s", c2kv_last_error(split.ctx));
        CHECK(fake::launched("attn_solo_kernel"), "splits that are asked for are the tensor cores'");
    }
    for (int tokens : {8, 30, 700}) {                             // and short chunks' extraction
        fake::launches.clear();
        CHECK(one.extract(tokens, 4) == C2KV_OK, "%s", c2kv_last_error(one.ctx));
        CHECK(fake::launched("attn_solo_kernel") == (tokens == 700) && fake::launched("extract_attn_kernel") != (tokens == 700),
              "%d tokens", tokens);
    }
}

}  // namespace

int main(int argc, char** argv) {
    const std::string name = argc > 1 ? argv[1] : "";
    if (name == "kernels") {
        for (const std::string& k : fake::kernel_names()) std::printf("%s\n", k.c_str());
        return 0;
    }
    if (name == "registers") registers(argv[2]);
    else if (name == "second_device") second_device();
    else if (name == "few_rows") few_rows();
    else if (name == "short64") short64();
    else if (name == "no_partials") no_partials();
    else if (name == "no_queries") no_queries();
    else CHECK(false, "unknown scenario '%s'", name.c_str());
    std::printf("ok\n");
}
