// Device tables of a plan on their way from host vectors to the device.  Small ones are collected into one allocation and
// one copy (twenty of each took most of the time of creating a small plan); a large one gets an allocation of its own.
//
// Lifetime: everything that is added belongs to the TableUpload until run().  A temporary or moved-in vector is kept, an
// lvalue is copied, so no vector of the caller has to outlive its add().
#pragma once
#include <cstddef>
#include <cstring>
#include <memory>
#include <type_traits>
#include <utility>
#include <vector>

namespace cqt {

class TableUpload {
  public:
    static constexpr size_t kSmall = 1 << 20;

    // dst is set by run(): the table's device address, null for an empty table
    template <class T>
    void add(T *&dst, std::vector<T> src) {
        static_assert(std::is_trivially_copyable<T>::value, "tables are copied byte by byte");
        dst = nullptr;
        const size_t n = src.size() * sizeof(T);
        if (n == 0) return;
        void **d = reinterpret_cast<void **>(&dst);
        if (n > kSmall) {
            auto kept = std::make_shared<std::vector<T>>(std::move(src));
            const void *data = kept->data();
            pieces_.push_back({d, std::shared_ptr<const void>(std::move(kept), data), 0, n});
            return;
        }
        const size_t off = (small_.size() + 255) / 256 * 256;
        small_.resize(off + n);
        std::memcpy(small_.data() + off, src.data(), n);
        pieces_.push_back({d, nullptr, off, n});
    }

    // upload(host, bytes, dev): allocates device memory, copies to it and sets dev; false: failed, no further table is set
    template <class Upload>
    bool run(Upload upload) {
        void *base = nullptr;
        if (!small_.empty() && !upload(static_cast<const void *>(small_.data()), small_.size(), base)) return false;
        for (Piece &p : pieces_) {
            void *own = static_cast<char *>(base) + p.offset;
            if (p.large && !upload(p.large.get(), p.bytes, own)) return false;
            *p.dst = own;
            p.large.reset();
        }
        return true;
    }

  private:
    struct Piece {
        void **dst;
        std::shared_ptr<const void> large;   // null: in small_, `offset` bytes from its start
        size_t offset, bytes;
    };
    std::vector<char> small_;
    std::vector<Piece> pieces_;
};

}  // namespace cqt
