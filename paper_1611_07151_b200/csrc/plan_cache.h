// Launch plans (tensor maps and kernel parameters) kept by the full request they were made for.
#pragma once

#include <cstddef>
#include <cstdint>
#include <cstring>
#include <memory>
#include <mutex>
#include <unordered_map>

#include "sqn.h"

namespace sqn {

// Key: plain data, every byte set (memset before filling).  A plan is handed out as a shared pointer: no copy (a plan is 2 KB)
// and safe when another thread's request empties the full cache.  Requests that no plan can serve are remembered too.
template <typename Key, typename Plan>
class PlanCache {
public:
    explicit PlanCache(size_t limit) : limit_(limit) {}

    // The plan for `key`, made by build(Plan*) -> status on the first request.
    template <typename Build>
    int get(const Key& key, std::shared_ptr<const Plan>* out, Build build)
    {
        {
            std::lock_guard<std::mutex> lock(mu_);
            auto it = plans_.find(key);
            if (it != plans_.end()) {
                *out = it->second;
                return *out ? SQN_OK : SQN_ERR_UNSUPPORTED;
            }
        }
        auto plan = std::make_shared<Plan>();
        const int rc = build(plan.get());
        if (rc != SQN_OK && rc != SQN_ERR_UNSUPPORTED) return rc;
        *out = rc == SQN_OK ? std::shared_ptr<const Plan>(std::move(plan)) : nullptr;
        std::lock_guard<std::mutex> lock(mu_);
        if (plans_.size() >= limit_) plans_.clear();
        plans_[key] = *out;
        return rc;
    }

private:
    struct Hash {
        size_t operator()(const Key& k) const
        {
            static_assert(sizeof(Key) % 8 == 0, "whole words");
            uint64_t w[sizeof(Key) / 8], h = 0x9e3779b97f4a7c15ull;
            std::memcpy(w, &k, sizeof(Key));
            for (uint64_t v : w) { h = (h ^ v) * 0xff51afd7ed558ccdull; h ^= h >> 32; }
            return (size_t)h;
        }
    };
    struct Equal {
        bool operator()(const Key& a, const Key& b) const { return std::memcmp(&a, &b, sizeof(Key)) == 0; }
    };
    std::mutex mu_;
    std::unordered_map<Key, std::shared_ptr<const Plan>, Hash, Equal> plans_;
    const size_t limit_;
};

}  // namespace sqn
