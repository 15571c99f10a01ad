// A recorded sequence of entry-point calls, issued from native code.  A training step launched call by call makes 14 to
// 160 of them, and through the binding each costs 10-15 us of host time (argument conversion, stream look-ups, views,
// events), several times what the launch itself takes: the device waits for the host.  Here one call issues them all
// with the same arguments on the same streams; nothing else about them changes.
#include <string.h>
#include <tuple>
#include <type_traits>
#include <utility>
#include "common.cuh"

namespace lpdt {

template <typename T>
static T word_to(uint64_t w) {
    if constexpr (std::is_pointer_v<T>) return reinterpret_cast<T>((uintptr_t)w);
    else if constexpr (std::is_same_v<T, float>) {
        const uint32_t b = (uint32_t)w;
        float f;
        memcpy(&f, &b, sizeof f);
        return f;
    } else return (T)(int64_t)w;
}

// f(words converted to its parameter types..., stream); the stream is every entry point's last parameter
template <typename... A, size_t... I>
static lpdt_status invoke(lpdt_status (*f)(A...), const uint64_t *w, void *stream, std::index_sequence<I...>) {
    using T = std::tuple<A...>;
    return f(word_to<std::tuple_element_t<I, T>>(w[I])..., stream);
}
template <auto F> struct Thunk;
template <typename... A, lpdt_status (*F)(A...)> struct Thunk<F> {
    static constexpr int kArgs = (int)sizeof...(A) - 1;
    static_assert(std::is_same_v<std::tuple_element_t<sizeof...(A) - 1, std::tuple<A...>>, void *>, "stream comes last");
    static lpdt_status run(const uint64_t *w, void *stream) {
        return invoke(F, w, stream, std::make_index_sequence<sizeof...(A) - 1>());
    }
};

struct Entry { const char *name; int args; lpdt_status (*run)(const uint64_t *, void *); };
#define LPDT_ENTRY(f) {#f, Thunk<f>::kArgs, Thunk<f>::run}
static const Entry kEntries[] = {
    LPDT_ENTRY(lpdt_fill_zero), LPDT_ENTRY(lpdt_quantize), LPDT_ENTRY(lpdt_quantize_with_range), LPDT_ENTRY(lpdt_quantize_batch),
    LPDT_ENTRY(lpdt_dequantize), LPDT_ENTRY(lpdt_qconv_fwd), LPDT_ENTRY(lpdt_qconv_bwd_data), LPDT_ENTRY(lpdt_qconv_bwd_weight),
    LPDT_ENTRY(lpdt_range_evonorm_fwd), LPDT_ENTRY(lpdt_range_evonorm_bwd), LPDT_ENTRY(lpdt_range_evonorm_fwd_q8),
    LPDT_ENTRY(lpdt_range_evonorm_bwd_q8), LPDT_ENTRY(lpdt_range_evonorm_pool_fwd),
    LPDT_ENTRY(lpdt_range_evonorm_pool_bwd), LPDT_ENTRY(lpdt_range_evonorm_bwd_params_batch), LPDT_ENTRY(lpdt_dequantize_acc_batch),
    LPDT_ENTRY(lpdt_gossip_mix), LPDT_ENTRY(lpdt_gossip_mix_q8), LPDT_ENTRY(lpdt_sgd_gossip_mix), LPDT_ENTRY(lpdt_sgd_update),
    LPDT_ENTRY(lpdt_residual_add), LPDT_ENTRY(lpdt_residual_add_bwd), LPDT_ENTRY(lpdt_avgpool), LPDT_ENTRY(lpdt_avgpool_bwd),
    LPDT_ENTRY(lpdt_maxpool2x2), LPDT_ENTRY(lpdt_maxpool2x2_bwd), LPDT_ENTRY(lpdt_softmax_ce), LPDT_ENTRY(lpdt_colsum)};
constexpr int kNumEntries = (int)(sizeof(kEntries) / sizeof(kEntries[0]));

}  // namespace lpdt

using namespace lpdt;

extern "C" int32_t lpdt_call_id(const char *name) {
    for (int i = 0; name && i < kNumEntries; ++i)
        if (!strcmp(kEntries[i].name, name)) return i;
    return -1;
}

extern "C" lpdt_status lpdt_run_calls(const uint64_t *code, int64_t n_words, void *const *streams, int32_t n_streams,
                                      int64_t *failed) {
    LPDT_CHECK_ARG(n_words >= 0 && (n_words == 0 || code) && n_streams >= 0 && (n_streams == 0 || streams));
    int64_t item = 0;
    for (int64_t i = 0; i < n_words; ++item) {
        if (failed) *failed = item;
        const int64_t id = (int64_t)code[i];
        if (id == LPDT_CALL_WAIT) {                       // stream b waits for what stream a holds so far, through an event
            LPDT_CHECK_ARG(i + 4 <= n_words && code[i + 1] < (uint64_t)n_streams && code[i + 2] < (uint64_t)n_streams && code[i + 3]);
            cudaEvent_t e = (cudaEvent_t)(uintptr_t)code[i + 3];
            LPDT_CUDA(cudaEventRecord(e, as_stream(streams[code[i + 2]])));
            LPDT_CUDA(cudaStreamWaitEvent(as_stream(streams[code[i + 1]]), e, 0));
            i += 4;
            continue;
        }
        LPDT_CHECK_ARG(id >= 0 && id < kNumEntries && i + 2 + kEntries[id].args <= n_words && code[i + 1] < (uint64_t)n_streams);
        const lpdt_status s = kEntries[id].run(code + i + 2, streams[code[i + 1]]);
        if (s != LPDT_OK) return s;
        i += 2 + kEntries[id].args;
    }
    return LPDT_OK;
}
